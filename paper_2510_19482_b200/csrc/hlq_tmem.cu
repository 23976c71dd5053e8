// Batches of more than ELUTQ_FRAGMENT_MAX_M rows at G = 128, but for those that hlq_mma.cu takes (rebuilds_in_shared_memory in
// api.cu): dequantise-and-contract on the 5th-generation tensor cores, the rebuilt weights as the A operand in TENSOR MEMORY.
//
// A rebuilt fp16 weight never passes through shared memory: a producer lane owns one weight row (= one TMEM lane), rebuilds
// 128 k of it in registers and stores them to its lane; the activations are the B operand, so the MMA's N is the batch and a
// small batch pays for no padding beyond 16 rows.
//
//   step       256 weight rows (two row blocks, UMMA M = 128 each) x 128 k x one token tile of up to 128 rows.  The two
//              blocks share the activation tile, which is what the L2 has to feed again and again.  The steps of a call,
//              tile by tile, are dealt to the CTAs (one per SM) in equal contiguous runs, so no SM idles for a wave.  The
//              parts of a tile that several CTAs share go to the workspace and are added in ascending k order (bit-reproducible)
//              by the CTA that comes last or, where there are many, by a second kernel.  Or the CTAs of a cluster share the K of a
//              tile and add up through their shared memory (a rule on costs: plan_of).
//   warps      0 weight loader (one bulk copy per row block and 512 k: eight packed tiles, contiguous in the blob), 1 MMA issuer, 2 activation loader
//              (TMA, 128-byte swizzle; few tokens: 2 and 3, by loads and stores, in another order), 4-19 producers: two warpgroups per row block, which take
//              the steps in turn, rebuild the weights, and at the end of a tile write out half of its tokens each.  (Four warps
//              per scheduler: with two, the latencies of a step's parameters, waits and stores were half of the time.)
//   slot       one 128-k step of one row block: 64 TMEM columns above the accumulators (2 x tokens columns).
//   dequant    W_hat = z + sum_j b_j s_j: a byte of plane j (8 weights) is copied to positions 8..15 of both halves of a word;
//              one logic operation leaves the bits of one weight pair, which read as fp16 are powers of two (at position 15 a
//              sign), and one packed fma multiplies with the scale over that power and adds: 3.5 half-rate or full-rate issue
//              slots per pair and plane.  (Moving the bits to the sign positions by a multiplication, an xor with s_j / 2 and an add: 5.5.)
//              Few tokens (PERM): k and k + 16 of the activations side by side, as the two halves of a word of weight bits lie.  A word shifted (by a
//              multiplication, but for one in four) has four bits of each half at positions 11 to 14; no byte permute, no sign.
//
//   bound      the producers' integer logic pipe (q = 4: 320 of a slot's 470 operations are the dequantisation itself, 65 to 75 % of
//              the pipe's cycles); from 96 tokens also the activations' way from the L2.  Against weights rebuilt in shared memory with one
//              barrier per step, us: 57344 x 8192, q = 4, M = 64 277 -> 145; 28672 x 4096, q = 2, M = 32 / 128 / 384
//              49 / 51 / 110 -> 25 / 33 / 95; 4096 x 14336, q = 3, M = 64 34 -> 24; 4096 x 4096, q = 2, M = 256 30 -> 18.
//
// Every wait is bounded; a thread whose wait runs out raises the status word and a CTA-wide flag that ends the other
// roles' waits; copies and MMAs in flight are waited for (bounded), tensor memory is freed, the kernel returns.
#include <cuda.h>

#include <initializer_list>
#include <mutex>

#include "common.cuh"

namespace elutq {

namespace {

constexpr int kCtrlWarps = 4, kBlocks = 2, kTurns = 2;         // row blocks; warpgroups per row block
constexpr int kTmThreads = 32 * (kCtrlWarps + 4 * kBlocks * kTurns);
constexpr int kBlockRows = 128;                 // weight rows per block (UMMA M)
constexpr int kTileRowsN = kBlocks * kBlockRows;
constexpr int kSlotCols = 64;                   // TMEM columns of a slot: 128 k of fp16 pairs
constexpr int kTmemCols = 512;
constexpr int kMaxTokens = 128;                 // tokens per tile (UMMA N)
constexpr uint32_t kTmWaitLimit = 1u << 20, kPollNs = 60;
constexpr int kMaxSplit = 8;                    // CTAs of a cluster
constexpr int kMaxX = 8, kMaxW = 4, kMaxSlots = 3;

struct TmemArgs {
    GemmArgs g;
    int mp, m_tiles;            // tokens per tile (a multiple of 16), token tiles
    int n_steps;                // 128-k steps of the whole K: steps of a tile
    int tile0;                  // first tile of this launch (0 but for clusters)
    int steps, per_cta;         // all steps; steps of one CTA
    int split;                  // CTAs of a cluster, which share a tile's K (1: no cluster)
    int reduce;                 // the CTAs add the parts of shared tiles themselves
    int exchange;               // cluster: where in shared memory the parts of a tile meet (0: over the rings, once these have been read)
    int xs, ws, ss;             // ring lengths: activation steps, weight chunks and slots (of a row block)
};

// mbarriers, in order; weights and slots have one ring per row block, accumulators one barrier each
enum { kBarWFull = 0, kBarWEmpty = kBarWFull + kBlocks * kMaxW, kBarXFull = kBarWEmpty + kBlocks * kMaxW, kBarXEmpty = kBarXFull + kMaxX,
       kBarAFull = kBarXEmpty + kMaxX, kBarAEmpty = kBarAFull + kBlocks * kMaxSlots, kBarDFull = kBarAEmpty + kBlocks * kMaxSlots,
       kBarDEmpty = kBarDFull + kBlocks, kBarDrain = kBarDEmpty + kBlocks, kNumBars };
constexpr int kMaxSmem = 232448, kFixed = kNumBars * 8 + 64;   // dynamic shared memory; of it barriers and flags

template <int Q>
struct TmCfg {
    static constexpr int PLANE_BYTES = 1024 * Q;
    static constexpr int TILE_BYTES = PLANE_BYTES + 128 * (Q + 1);
    static constexpr int UNIT_BYTES = 8 * TILE_BYTES;         // 512 k of one row block
};

__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ uint64_t sw128_desc(uint32_t saddr) {       // K-major, 128-byte swizzle, 1024 bytes per 8 rows
    return (uint64_t)((saddr >> 4) & 0x3FFFu) | ((uint64_t)1 << 16) | ((uint64_t)(1024u >> 4) << 32) | ((uint64_t)1 << 46) |
           ((uint64_t)2 << 61);
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" :: "r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_expect(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" :: "r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                 : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    return ok != 0;
}
__device__ __forceinline__ void commit_to(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" :: "r"(bar) : "memory");
}
__device__ __forceinline__ void mma_ts(uint32_t d, uint32_t a, uint64_t b, uint32_t idesc, uint32_t accumulate) {
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\ttcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
                 :: "r"(d), "r"(a), "l"(b), "r"(idesc), "r"(accumulate) : "memory");
}
// True in one lane of the (converged) warp.  The condition around tcgen05 instructions has to be this alone: only then does the
// compiler know that one lane issues them, and an MMA takes about 10 cycles to issue; otherwise it takes 50 to 90.
__device__ __forceinline__ bool elect_one() {
    uint32_t e;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(e));
    return e != 0;
}
__device__ __forceinline__ void tmem_st16(uint32_t addr, const uint32_t (&r)[16]) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};"
                 :: "r"(addr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]),
                 "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]) : "memory");
}
__device__ __forceinline__ void tmem_st8(uint32_t addr, const uint32_t* r) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};"
                 :: "r"(addr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]) : "memory");
}
__device__ __forceinline__ void tmem_ld16(uint32_t (&r)[16], uint32_t addr) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
                   "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
                 : "r"(addr) : "memory");
}
__device__ __forceinline__ void tmem_ld_wait(uint32_t (&r)[16]) {     // names the registers: nothing may use them earlier
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
                   "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15]) :: "memory");
}

// slot and parity of the n-th use of a ring, advanced without divisions
struct Ring {
    int len, i;
    uint32_t phase;
    __device__ __forceinline__ Ring(int n) : len(n), i(0), phase(0) {}
    __device__ __forceinline__ void next() {
        if (++i == len) { i = 0; phase ^= 1u; }
    }
};

// The run of steps of a CTA, cut at the ends of tiles and of 512-k chunks.
struct Walk {
    int t, t1, n_steps, tile, step, end;                      // steps [step, end) of the tile are next
    bool first;
    __device__ __forceinline__ Walk(int t0, int t1_, int n) : t(t0), t1(t1_), n_steps(n), tile(t0 / n), step(t0 - tile * n), first(true) { cut(); }
    __device__ __forceinline__ void cut() { end = min(min((step | 3) + 1, n_steps), step + (t1 - t)); }
    __device__ __forceinline__ bool more() const { return t < t1; }
    __device__ __forceinline__ bool begins() const { return first || step == 0; }                 // a new accumulation
    __device__ __forceinline__ bool ends() const { return end == n_steps || t + (end - step) == t1; }
    __device__ __forceinline__ void next() {
        t += end - step;
        step = end;
        first = false;
        if (step == n_steps) { step = 0; ++tile; }
        cut();
    }
};

// A constant that the compiler keeps in a register (one logic operation takes a single immediate).
__device__ __forceinline__ uint32_t opaque(uint32_t v) {
    asm volatile("mov.b32 %0, %0;" : "+r"(v));
    return v;
}

// How many warps before this one took the ticket: read, or (add = 1 and a mark) announced behind the warp's own writes.
__device__ __forceinline__ unsigned ticket_seen(unsigned* ticket, int lane, unsigned add) {
    unsigned t = 0;
    __syncwarp();
    if (lane == 0) {
        if (add) asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], %2;" : "=r"(t) : "l"(ticket), "r"(add) : "memory");
        else asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(t) : "l"(ticket) : "memory");
    }
    __syncwarp();                                              // lane 0 has acquired for the whole warp (a shuffle orders no memory)
    return __shfl_sync(0xffffffffu, t, 0);
}

__device__ __forceinline__ __half2 as_half2(uint32_t v) { return *reinterpret_cast<const __half2*>(&v); }

// CLUSTER: a tile's K is shared by the CTAs of a cluster.  PERM > 0: that many tokens, whose activations are put in the order of a word's halves.
template <int Q, bool CLUSTER, int PERM>
__global__ void __launch_bounds__(kTmThreads, 1) hlq_tmem_kernel(const __grid_constant__ CUtensorMap xmap, const TmemArgs a) {
    using C = TmCfg<Q>;
    extern __shared__ __align__(1024) uint8_t smem[];
    const int blk_bytes = a.mp * 128;                         // activations of 64 k
    const int x_bytes = 2 * blk_bytes;                        // one step
    uint8_t* sX = smem;
    uint8_t* sW = sX + a.xs * x_bytes;
    uint64_t* bars = reinterpret_cast<uint64_t*>(sW + kBlocks * a.ws * C::UNIT_BYTES);
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + kNumBars);
    volatile uint32_t* give_up = tmem_slot + 1;
    const uint32_t bar0 = smem_addr(bars);
    auto bar = [&](int i) { return bar0 + 8u * (uint32_t)i; };

    const int tid = threadIdx.x, lane = tid & 31;
    const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);   // warp-uniform for the compiler too
    uint4 h0;
    uint2 h1;
    blob_header_load(a.g.tiles, h0, h1);
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" :: "r"(smem_addr(tmem_slot)), "n"(kTmemCols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (CLUSTER && a.exchange != 0) cluster_arrive();          // (this CTA is there: awaited before its peers write to it)
    if (tid == 0) {
        auto init = [&](int i, int n) { asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" :: "r"(bar(i)), "r"(n) : "memory"); };
        for (int i = 0; i < kBlocks * kMaxW; ++i) { init(kBarWFull + i, 1); init(kBarWEmpty + i, 4 * kTurns); }
        for (int i = 0; i < kMaxX; ++i) { init(kBarXFull + i, PERM > 16 ? 2 : 1); init(kBarXEmpty + i, 1); }
        for (int i = 0; i < kBlocks * kMaxSlots; ++i) { init(kBarAFull + i, 4); init(kBarAEmpty + i, 1); }
        for (int i = 0; i < kBlocks; ++i) { init(kBarDFull + i, 1); init(kBarDEmpty + i, 4 * kTurns); }
        init(kBarDrain, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        *give_up = 0;
        asm volatile("prefetch.tensormap [%0];" :: "l"(&xmap) : "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = *tmem_slot;
    const uint32_t slot_col0 = (uint32_t)(kTmemCols - kBlocks * a.ss * kSlotCols);   // accumulators below, slots above

    const int b = blockIdx.x, base_tile = CLUSTER ? a.tile0 : 0;
    int t0 = b * a.per_cta, t1 = min(a.steps, t0 + a.per_cta);
    if constexpr (CLUSTER) {
        const int tile = b / a.split, r = b - tile * a.split;
        t0 = tile * a.n_steps + a.n_steps * r / a.split;
        t1 = tile * a.n_steps + a.n_steps * (r + 1) / a.split;
    }
    if (!blob_header_ok(h0, h1, Q, 128, a.g.N, a.g.K)) {      // before any tile is read; the same answer in every thread: no work
        t1 = t0;
        if (tid == 0 && a.g.counters != nullptr) atomicExch(a.g.counters, kStatusBlobMismatch);
    }
    [[maybe_unused]] bool have_part = false;                 // CLUSTER: this warp's sums are in tensor memory
    const uint32_t limit = a.g.wait_limit ? a.g.wait_limit : kTmWaitLimit;

    // Bounded wait; false once this CTA has given up.  (Sleeping between polls: the waiting warps' instructions cost the
    // producers 3 to 8 %, whatever the length.)  What has to be waited for may hang on the kernel before this one, which the limit
    // is not to time.
    auto wait = [&](int i, uint32_t parity) {
        if (mbar_try(bar(i), parity)) return true;
        grid_dependency_wait();
        for (uint32_t n = 0; n < limit; ++n) {
            __nanosleep(kPollNs);
            if (mbar_try(bar(i), parity)) return true;
            if ((n & 15u) == 15u && *give_up) return false;
        }
        *give_up = 1;
        if (a.g.counters != nullptr) atomicExch(a.g.counters, kStatusWaitExpired);
        return false;
    };
    auto wait_warp = [&](int i, uint32_t parity) { return __all_sync(0xffffffffu, wait(i, parity)) != 0; };
    // A loader's copies land before its CTA may leave (or a peer write into its shared memory), whoever gave up: a loader that has
    // issued everything does not notice that the others did.
    auto drain = [&](int bar_full, int len, int issued) {
        for (int n = max(0, issued - len); n < issued; ++n)
            for (uint32_t t = 0; t < kTmWaitLimit && !mbar_try(bar(bar_full + n % len), (uint32_t)(n / len) & 1u); ++t) {}
    };

    if (warp == 0) {
        // ---- weight loader (weights do not depend on the previous kernel) ----------------------------------------------------------
        grid_launch_dependents();
        if (lane == 0) {
            Ring w(a.ws);
            int issued[kBlocks] = {};
            bool ok = true;
            for (Walk r(t0, t1, a.n_steps); r.more() && ok; r.next()) {
                for (int blk = 0; blk < kBlocks; ++blk) {
                    ok = wait(kBarWEmpty + blk * kMaxW + w.i, w.phase ^ 1u);
                    if (!ok) break;
                    const int rb0 = ((r.tile + base_tile) / a.m_tiles) * (kBlocks * 8) + blk * 8, nrb = max(0, min(8, a.g.n_rb - rb0));
                    const uint32_t bytes = (uint32_t)(nrb * C::TILE_BYTES), mb = bar(kBarWFull + blk * kMaxW + w.i);
                    mbar_expect(mb, bytes);
                    if (nrb > 0)
                        asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                                     :: "r"(smem_addr(sW) + (uint32_t)((blk * a.ws + w.i) * C::UNIT_BYTES)),
                                        "l"(a.g.tiles + ((size_t)(r.step >> 2) * a.g.n_rb + rb0) * C::TILE_BYTES), "r"(bytes), "r"(mb) : "memory");
                    ++issued[blk];
                }
                w.next();
            }
            for (int blk = 0; blk < kBlocks; ++blk) drain(kBarWFull + blk * kMaxW, a.ws, issued[blk]);
        }
    } else if (PERM > 0 && (warp == 2 || warp == 3)) {
        // ---- activation loaders of few tokens: a lane takes 32 k of a token and puts k and k + 16 side by side, as the two halves of a word of weight
        // bits lie.  16 tokens: the two warps take the steps in turn; 32: half of the tokens of every step each, with the loads of two steps on their way, so that
        // a step waits for half as many (in turn 1 to 5 % slower, us, q = 1 and 2, M = 32: 28672 x 4096 22.0 and 25.5, now 21.5 and 24.8; 37888 x 2048, q = 2 16.6, now
        // 16.3).  (Walking instead of dividing: M = 32 3 to 5 % faster, since the divisions take the rebuild's pipes.) ------------
        grid_dependency_wait();
        constexpr bool kHalves = PERM > 16;
        constexpr int kGroups = 2, kDeep = kHalves ? 2 : 1, kStride = kHalves ? 1 : 2;      // groups of 8 tokens, steps on their way
        const int first = kHalves ? 0 : warp - 2, m_lane = lane >> 2, c = lane & 3, m0 = (kHalves ? (warp - 2) * 16 : 0) + m_lane;
        const __half* x = a.g.X + (size_t)m0 * a.g.K + c * 32;       // (one token tile: step t is step t mod n_steps of K)
        const uint32_t at = (uint32_t)((c >> 1) * blk_bytes + m0 * 128 + ((4 * (c & 1) ^ m_lane) << 4));
        int step = t0 % a.n_steps, left = t1 - t0 - first, slot = first;
        uint32_t phase = 0;
        uint4 v[kDeep][kGroups][4];
        auto on = [&](int by) {
            step += by;
            while (step >= a.n_steps) step -= a.n_steps;
        };
        auto fetch = [&](uint4 (&r)[kGroups][4], bool more) {
            const __half* xk = x + step * 128;
#pragma unroll
            for (int g = 0; g < kGroups; ++g) {
                const bool there = more && m0 + 8 * g < a.g.M;
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    r[g][e] = there ? reinterpret_cast<const uint4*>(xk + (size_t)(8 * g) * a.g.K)[e] : make_uint4(0, 0, 0, 0);
            }
            on(kStride);
        };
        on(first);
#pragma unroll
        for (int d = 0; d < kDeep; ++d) fetch(v[d], left > d * kStride);
        for (bool ok = true; ok && left > 0;) {
#pragma unroll
            for (int d = 0; d < kDeep; ++d) {
                if (left <= 0) break;
                ok = wait_warp(kBarXEmpty + slot, phase ^ 1u);
                if (!ok) break;
                uint8_t* dst = sX + slot * x_bytes;
#pragma unroll
                for (int g = 0; g < kGroups; ++g) {
#pragma unroll
                    for (int e = 0; e < 2; ++e) {             // bytes e and e + 2 of the words
                        const uint4 lo = v[d][g][e], hi = v[d][g][e + 2];
                        const uint4 o[2] = {make_uint4(__byte_perm(lo.x, hi.x, 0x5410), __byte_perm(lo.x, hi.x, 0x7632), __byte_perm(lo.y, hi.y, 0x5410), __byte_perm(lo.y, hi.y, 0x7632)),
                                            make_uint4(__byte_perm(lo.z, hi.z, 0x5410), __byte_perm(lo.z, hi.z, 0x7632), __byte_perm(lo.w, hi.w, 0x5410), __byte_perm(lo.w, hi.w, 0x7632))};
#pragma unroll
                        for (int i = 0; i < 2; ++i) *reinterpret_cast<uint4*>(dst + (at ^ ((2 * e + i) << 4)) + g * 1024) = o[i];
                    }
                }
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                __syncwarp();
                if (lane == 0) mbar_arrive(bar(kBarXFull + slot));
                left -= kStride;
                fetch(v[d], left > (kDeep - 1) * kStride);
                slot += kStride;
                if (slot >= a.xs) {
                    slot -= a.xs;
                    phase ^= 1u;
                }
            }
        }
    } else if (warp == 2) {
        // ---- activation loader: a step is two boxes of 64 k ------------------------------------------------------------------
        grid_dependency_wait();
        if (lane == 0) {
            Ring x(a.xs);
            int issued = 0;
            bool ok = true;
            for (Walk r(t0, t1, a.n_steps); r.more() && ok; r.next()) {
                const int m0 = ((r.tile + base_tile) % a.m_tiles) * a.mp;
                for (int step = r.step; step < r.end; ++step) {
                    ok = wait(kBarXEmpty + x.i, x.phase ^ 1u);
                    if (!ok) break;
                    const uint32_t dst = smem_addr(sX) + (uint32_t)(x.i * x_bytes), mb = bar(kBarXFull + x.i);
                    mbar_expect(mb, (uint32_t)x_bytes);
                    for (int kb = 0; kb < 2; ++kb)
                        asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
                                     :: "r"(dst + (uint32_t)(kb * blk_bytes)), "l"(&xmap), "r"(step * 128 + kb * 64), "r"(m0), "r"(mb) : "memory");
                    ++issued;
                    x.next();
                }
            }
            drain(kBarXFull, a.xs, issued);
        }
    } else if (warp == 1) {
        // ---- MMA issuer: one elected lane ------------------------------------------------------------------------------------
        const int last = test_stalls(a.g.flags) ? t0 : t1;   // (test flag: nothing is issued or completes, the waits run out)
        if (elect_one()) {
            const uint32_t idesc = (1u << 4) | ((uint32_t)(a.mp >> 3) << 17) | ((uint32_t)(kBlockRows >> 4) << 24);
            const uint64_t x_desc0 = sw128_desc(smem_addr(sX));
            const uint32_t x_units = (uint32_t)x_bytes >> 4, blk_units = (uint32_t)blk_bytes >> 4;
            Ring x(a.xs), s(a.ss);
            uint32_t d_phase = 1;
            bool live = true;
            for (Walk r(t0, last, a.n_steps); r.more() && live; r.next()) {
                for (int step = r.step; step < r.end && live; ++step) {
                    const bool begins = r.begins() && step == r.step, ends = r.ends() && step == r.end - 1;
                    const uint64_t b0 = x_desc0 + (uint64_t)((uint32_t)x.i * x_units), b1 = b0 + blk_units;
#pragma unroll
                    for (int blk = 0; blk < kBlocks; ++blk) {
                        if (blk == 0) live = wait(kBarXFull + x.i, x.phase);
                        if (begins && live) live = wait(kBarDEmpty + blk, d_phase);
                        if (live) live = wait(kBarAFull + blk * kMaxSlots + s.i, s.phase);
                        if (!live) break;
                        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                        const uint32_t acc = tmem + (uint32_t)(blk * a.mp);
                        const uint32_t at = tmem + slot_col0 + (uint32_t)((blk * a.ss + s.i) * kSlotCols);
#pragma unroll
                        for (int kk = 0; kk < 8; ++kk)
                            mma_ts(acc, at + 8u * kk, (kk < 4 ? b0 : b1) + (uint64_t)((kk & 3) * 2), idesc, (kk == 0 && begins) ? 0u : 1u);
                        commit_to(bar(kBarAEmpty + blk * kMaxSlots + s.i));
                        if (blk == kBlocks - 1) commit_to(bar(kBarXEmpty + x.i));
                        if (ends) commit_to(bar(kBarDFull + blk));
                    }
                    x.next();
                    s.next();
                    if (begins) d_phase ^= 1u;
                }
            }
            // everything issued has completed before tensor memory is freed
            commit_to(bar(kBarDrain));
            for (uint32_t t = 0; t < kTmWaitLimit && !mbar_try(bar(kBarDrain), 0); ++t) {}
        }
        __syncwarp();
    } else if (warp >= kCtrlWarps) {
        // ---- producers ---------------------------------------------------------------------------------------------------------
        const int blk = ((warp - kCtrlWarps) >> 2) & 1, turn = (warp - kCtrlWarps) >> 3, quad = warp & 3;
        const int l = lane & 15, item = 2 * quad + (lane >> 4);
        const int word_rot = l >> 2, byte_rot = (l & 3) * 8;   // the packed layout rotates a row's 16 bytes by the row
        const uint32_t plane_mask = (a.g.flags & ELUTQ_FLAG_OFFSET_ONLY) ? 0u : 0xffffffffu;
        const uint32_t offset_mask = (a.g.flags & ELUTQ_FLAG_SKIP_OFFSET) ? 0u : 0xffffffffu;
        const uint32_t dst0 = tmem + slot_col0 + (uint32_t)(blk * a.ss * kSlotCols) + ((uint32_t)(quad * 32) << 16);
        const uint32_t pair3_mask = opaque(0x80004000u);
        Ring w(a.ws), s(a.ss);
        if (turn) s.next();
        uint32_t d_phase = 0;
        bool live = true;
        const size_t n_pad = (size_t)a.g.n_rb * kTileRows;
        const int M = a.g.M, N = a.g.N;
        const uint32_t acc = tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)(blk * a.mp);
        auto row_of = [&](int tile) { return ((tile + base_tile) / a.m_tiles) * kTileRowsN + blk * kBlockRows + quad * 32 + lane; };
        auto put16 = [&](int m, int n, int count, const uint32_t (&v)[16]) {
            if (!(a.g.flags & (ELUTQ_FLAG_OUT_F32 | ELUTQ_FLAG_ACCUMULATE))) {
                __half* y = reinterpret_cast<__half*>(a.g.Y) + (size_t)m * N + n;      // (one address that walks: see kStoreEights)
#pragma unroll
                for (int i = 0; i < 16; ++i)
                    if (i < count) { *y = __float2half_rn(__uint_as_float(v[i])); y += N; }
            } else {
#pragma unroll
                for (int i = 0; i < 16; ++i)
                    if (i < count) store_out(a.g, (size_t)(m + i) * N + n, __uint_as_float(v[i]));
            }
        };
        // Tickets of a shared tile, one per warp of the CTA: how many other parts are in the workspace; says that this warp's
        // is there now and whether it is the last.
        auto parts_of = [&](int tile) { return (tile * a.n_steps + a.n_steps - 1) / a.per_cta - tile * a.n_steps / a.per_cta + 1; };
        auto ticket_of = [&](int tile) { return a.g.tickets + tile * a.n_steps / a.per_cta * (4 * kBlocks * kTurns) + (warp - kCtrlWarps); };
        auto announce = [&](int tile, unsigned mark) {
            const unsigned t = ticket_seen(ticket_of(tile), lane, 1u + mark), last = (unsigned)(parts_of(tile) - 1);
            if ((t & (kTicketNoPart - 1)) == last && t + mark != last && lane == 0) *ticket_of(tile) = 0;     // parts are missing: nobody adds up
            return t + mark == last;
        };
        int head = -1, tail = -1;                              // shared tiles to add up, to finish
        Walk r(t0, t1, a.n_steps);
        for (; r.more() && live; r.next()) {
            live = wait_warp(kBarWFull + blk * kMaxW + w.i, w.phase);
            if (!live) break;
            const uint8_t* rec = sW + (blk * a.ws + w.i) * C::UNIT_BYTES + item * C::TILE_BYTES + l * 16;      // this row's packed tile
            auto release = [&]() {
                __syncwarp();
                if (lane == 0) mbar_arrive(bar(kBarWEmpty + blk * kMaxW + w.i));
            };
            int step = r.step + ((turn - (r.t - t0)) & 1);     // this warpgroup's turns
            if (step >= r.end) release();
#pragma unroll 1
            for (; step < r.end; step += 2) {
                const int h = step & 1, uu = (step >> 1) & 1;
                // the row's 16 plane bytes of the step in column order
                uint32_t pw[Q][4];
#pragma unroll
                for (int j = 0; j < Q; ++j) {
                    const uint8_t* v = rec + ((uu * Q + j) * 32 + 16 * h) * 16;
                    uint32_t t[4];
#pragma unroll
                    for (int i = 0; i < 4; ++i) t[i] = *reinterpret_cast<const uint32_t*>(v + ((i - word_rot) & 3) * 4);
#pragma unroll
                    for (int i = 0; i < 4; ++i) pw[j][i] = __funnelshift_l(t[(i + 3) & 3], t[i], byte_rot);
                }
                __half2 factor[Q][4], z2, start3;
                int down;
                bool any_up;
                // Its parameters s_0 .. s_{Q-1}, z, two to a word.  Plane j's bit at position 11 .. 14 of a half is 2^-13, 2^-11, 2^-7, 2 as an fp16
                // number, so that with factor[j][position] it contributes s_j (exact products).  Scales of 1 and more would not fit the factors:
                // such a row is built 2^-down times its size (down = exponent of its largest scale, plus one) and scaled up at the end.
                if constexpr (PERM > 0) {
                    uint32_t sc[Q / 2 + 1];
#pragma unroll
                    for (int i = 0; i <= Q / 2; ++i)
                        sc[i] = *reinterpret_cast<const uint32_t*>(rec + C::PLANE_BYTES - l * 12 + h * 64 + (uu * ((Q + 1) / 2) + i) * 128);
                    if (Q % 2 == 0) {                         // (an odd number of them: the second step's begin in the middle of a word)
#pragma unroll
                        for (int i = 0; i <= Q / 2; ++i) sc[i] = __funnelshift_r(sc[i], i < Q / 2 ? sc[i + 1] : 0u, uu * 16);
                    }
                    if (a.g.flags & (ELUTQ_FLAG_OFFSET_ONLY | ELUTQ_FLAG_SKIP_OFFSET)) {
#pragma unroll
                        for (int j = 0; j <= Q; ++j)
                            if (a.g.flags & (j < Q ? ELUTQ_FLAG_OFFSET_ONLY : ELUTQ_FLAG_SKIP_OFFSET)) sc[j / 2] &= j & 1 ? 0x0000ffffu : 0xffff0000u;
                    }
                    if (step + 2 >= r.end) release();
                    auto param = [&](int j) { return j & 1 ? __high2half2(as_half2(sc[j / 2])) : __low2half2(as_half2(sc[j / 2])); };
                    __half2 most = __habs2(param(0));
#pragma unroll
                    for (int j = 1; j < Q; ++j) most = __hmax2(most, __habs2(param(j)));
                    any_up = __any_sync(0xffffffffu, __low2float(most) >= 1.f);
                    __half2 down2 = __float2half2_rn(1.f);
                    z2 = param(Q);
                    down = 0;
                    if (any_up) {
                        down = max((int)(__half_as_ushort(__low2half(most)) >> 10) - 14, 0);
                        down2 = __float2half2_rn(__int_as_float((127 - down) << 23));          // exact, 2^-16 as a subnormal
                        z2 = __hmul2(z2, down2);
                    }
#pragma unroll
                    for (int j = 0; j < Q; ++j) {
                        const __half2 s2 = any_up ? __hmul2(param(j), down2) : param(j);
                        factor[j][0] = __hmul2(s2, __float2half2_rn(8192.f));
                        factor[j][1] = __hmul2(s2, __float2half2_rn(2048.f));
                        factor[j][2] = __hmul2(s2, __float2half2_rn(128.f));
                        factor[j][3] = __hmul2(s2, __float2half2_rn(0.5f));
                    }
                } else {
                // Its parameters s_0 .. s_{Q-1}, z.  Plane j's bit at position 8..14 of a half is 2^-16, 2^-15, 2^-14, 2^-13, 2^-11, 2^-7,
                // 2 as an fp16 number and at position 15 a sign, so that with factor[j][p] it contributes s_j (exact products),
                // as a sign +-s_j/2.  Scales of 1 and more would not fit the factors: such a row is built 2^-down times its
                // size (down = exponent of its largest scale, plus one) and scaled up at the end.
                uint32_t sc[Q + 1];                            // packed twice
                auto load_params = [&](auto uu_c) {
#pragma unroll
                    for (int c = 0; c <= Q; ++c) {
                        const int e = decltype(uu_c)::value * (Q + 1) + c;
                        sc[c] = *reinterpret_cast<const uint16_t*>(rec + C::PLANE_BYTES - l * 12 + h * 64 + (e >> 1) * 128 + (e & 1) * 2);
                    }
                };
                if (uu) load_params(IntC<1>{});
                else load_params(IntC<0>{});
                uint32_t top = 0;
#pragma unroll
                for (int c = 0; c <= Q; ++c) {
                    sc[c] = __byte_perm(sc[c] & (c == Q ? offset_mask : plane_mask), 0u, 0x1010);
                    if (c < Q) top = max(top, sc[c] & 0x7c00u);
                }
                if (step + 2 >= r.end) release();
                down = max((int)(top >> 10) - 14, 0);
                any_up = __any_sync(0xffffffffu, down != 0);
                z2 = as_half2(sc[Q]);
                float zhat = __low2float(z2);
#pragma unroll
                for (int j = 0; j < Q; ++j) zhat += 0.5f * __low2float(as_half2(sc[j]));
                __half2 zh2 = __float2half2_rn(zhat);
                if (any_up) {
                    const __half2 down2 = __float2half2_rn(__int_as_float((127 - down) << 23));        // exact, 2^-16 as a subnormal
                    z2 = __hmul2(z2, down2);
                    zh2 = __hmul2(zh2, down2);
#pragma unroll
                    for (int j = 0; j < Q; ++j) {
                        const __half2 t = __hmul2(as_half2(sc[j]), down2);
                        sc[j] = *reinterpret_cast<const uint32_t*>(&t);
                    }
                }
#pragma unroll
                for (int j = 0; j < Q; ++j) {
                    const __half2 s2 = as_half2(sc[j]);
                    factor[j][0] = __hmul2(__hmul2(s2, __floats2half2_rn(8192.f, 4096.f)), __float2half2_rn(8.f));
                    factor[j][1] = __hmul2(s2, __floats2half2_rn(16384.f, 8192.f));
                    factor[j][2] = __hmul2(s2, __floats2half2_rn(2048.f, 128.f));
                    factor[j][3] = __hmul2(s2, __float2half2_rn(0.5f));
                }
                start3 = __lows2half2(z2, zh2);  // weight 7 of a byte has its bit at the sign
                }

                live = wait_warp(kBarAEmpty + blk * kMaxSlots + s.i, s.phase ^ 1u);
                if (!live) break;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint32_t dst = dst0 + (uint32_t)(s.i * kSlotCols);
                auto scale_up = [&](auto& r, int from = 0, int to = 16) {
                    const __half2 up0 = __float2half2_rn(__int_as_float((127 + (down >> 1)) << 23));
                    const __half2 up1 = __float2half2_rn(__int_as_float((127 + ((down + 1) >> 1)) << 23));
#pragma unroll
                    for (int i = 0; i < 16; ++i) {
                        if (i < from || i >= to) continue;
                        const __half2 t = __hmul2(__hmul2(as_half2(r[i]), up0), up1);
                        r[i] = *reinterpret_cast<const uint32_t*>(&t);
                    }
                };
                // Registers are short: at q = 4 sixteen rebuilt words at a time and an address for every token written out spilled, and a tile's end took 0.1
                // us for 16 and 0.4 for 32 tokens.  In eights, with one address (for all q and numbers of tokens): us, 19456 x 256, q = 4, M = 32 6.05 -> 5.59, M = 16 5.38 ->
                // 5.2, 37888 x 768, M = 32 13.4 -> 12.5; 28672 x 4096, M = 64, q = 3 34.8 -> 33.5, M = 128, q = 2 32.6 -> 31.6.  (Clusters of 32 tokens: eights spill.)
                constexpr bool kStoreEights = PERM > 0 && Q == 4 && !(CLUSTER && PERM > 16);
#pragma unroll
                for (int i4 = 0; i4 < 4; ++i4) {
                    uint32_t o[16];
                    if constexpr (PERM > 0) {
                        // 32 weights: register 8 e + i holds bit i of bytes e and e + 2
#pragma unroll
                        for (int v = 0; v < 4; ++v) {         // bits 0-3 and 4-7 of bytes 0 and 2, of bytes 1 and 3
                            __half2 acc[4] = {z2, z2, z2, z2};
#pragma unroll
                            for (int j = 0; j < Q; ++j) {
                                const uint32_t w = pw[j][i4], x = v == 0 ? w * 2048u : v == 1 ? w * 128u : v == 2 ? w * 8u : w >> 1;
#pragma unroll
                                for (int p = 0; p < 4; ++p) acc[p] = __hfma2(as_half2(x & (0x08000800u << p)), factor[j][p], acc[p]);
                            }
#pragma unroll
                            for (int p = 0; p < 4; ++p) o[4 * v + p] = *reinterpret_cast<const uint32_t*>(&acc[p]);
                            if constexpr (kStoreEights) {
                                if (v & 1) {
                                    if (any_up) scale_up(o, 4 * v - 4, 4 * v + 4);
                                    tmem_st8(dst + 16u * i4 + 4u * v - 4u, o + 4 * v - 4);
                                }
                            }
                        }
                    } else {
#pragma unroll
                    for (int by = 0; by < 4; ++by) {
                        __half2 acc[4] = {z2, z2, z2, start3};
#pragma unroll
                        for (int j = 0; j < Q; ++j) {
                            const uint32_t x = __byte_perm(pw[j][i4], 0u, 0x0404u | (uint32_t)(by * 0x1010));
#pragma unroll
                            for (int p = 0; p < 4; ++p) {
                                uint32_t t;
                                if (p < 3) t = x & ((0x0100u << (2 * p)) | (0x02000000u << (2 * p)));
                                else asm("lop3.b32 %0, %1, %2, 0xbc000000, 0x6a;" : "=r"(t) : "r"(x), "r"(pair3_mask));     // high half -1 or 1
                                acc[p] = __hfma2(as_half2(t), factor[j][p], acc[p]);
                            }
                        }
#pragma unroll
                        for (int p = 0; p < 4; ++p) o[4 * by + p] = *reinterpret_cast<const uint32_t*>(&acc[p]);
                    }
                    }
                    if constexpr (!kStoreEights) {
                        if (any_up) scale_up(o);
                        tmem_st16(dst + 16u * i4, o);
                    }
                }
                asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
                asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                __syncwarp();
                if (lane == 0) mbar_arrive(bar(kBarAFull + blk * kMaxSlots + s.i));
                s.next();
                s.next();
            }
            if (!live) break;
            w.next();
            if (r.ends()) {
                grid_dependency_wait();
                live = wait_warp(kBarDFull + blk, d_phase);
                if (!live) break;
                d_phase ^= 1u;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                // This warp's 32 rows and every other 16 tokens to Y, or to the workspace.  (A last part that its CTA adds up
                // itself: below.)
                const bool to_end = r.end == a.n_steps, whole = to_end && r.tile * a.n_steps >= t0;
                if (CLUSTER || (a.reduce && !to_end)) {
                    tail = r.tile;
                    break;
                }
                const int m0 = ((r.tile + base_tile) % a.m_tiles) * a.mp, m_count = min(a.mp, M - m0), n = row_of(r.tile);
                float* part = a.g.partials + ((size_t)(b - r.tile * a.n_steps / a.per_cta) * M + m0) * n_pad + n;
                for (int c0 = 16 * turn; c0 < m_count; c0 += 16 * kTurns) {
                    uint32_t v[16];
                    tmem_ld16(v, acc + (uint32_t)c0);
                    tmem_ld_wait(v);
                    const int mc = m_count - c0;
                    if (!whole) {
                        if ((size_t)n < n_pad) {
#pragma unroll
                            for (int i = 0; i < 16; ++i)
                                if (i < mc) part[(size_t)(c0 + i) * n_pad] = __uint_as_float(v[i]);
                        }
                    } else if (n < N) {
                        put16(m0 + c0, n, mc, v);
                    }
                }
                if (a.reduce && !whole && announce(r.tile, 0)) head = r.tile;
                asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                __syncwarp();
                if (lane == 0) mbar_arrive(bar(kBarDEmpty + blk));
            }
        }
        if constexpr (CLUSTER) have_part = live && tail >= 0;
        else {
            if (!live && a.reduce) {                           // the tickets not taken yet: of the run's first tile (once it ends), of its last
                grid_dependency_wait();
                const int first = t0 / a.n_steps, last = (t1 - 1) / a.n_steps;
                if (r.tile == first && parts_of(first) > 1) announce(first, kTicketNoPart);
                if (last != first && t1 < (last + 1) * a.n_steps) announce(last, kTicketNoPart);
            }
            // Shared tiles: the warp that finds all other parts in the workspace adds them to its own in ascending k order (no
            // warp waits for another; a tile's other parts are mostly those that their CTAs began with, long written).
            if (live && tail >= 0) {
                const int mine = b - tail * a.n_steps / a.per_cta, m0 = ((tail + base_tile) % a.m_tiles) * a.mp, m_count = min(a.mp, M - m0), n = row_of(tail);
                if (ticket_seen(ticket_of(tail), lane, 0) != (unsigned)(parts_of(tail) - 1)) {
                    float* part = a.g.partials + ((size_t)mine * M + m0) * n_pad + n;
                    for (int c0 = 16 * turn; c0 < m_count; c0 += 16 * kTurns) {
                        uint32_t v[16];
                        tmem_ld16(v, acc + (uint32_t)c0);
                        tmem_ld_wait(v);
#pragma unroll
                        for (int i = 0; i < 16; ++i)
                            if (c0 + i < m_count && (size_t)n < n_pad) part[(size_t)(c0 + i) * n_pad] = __uint_as_float(v[i]);
                    }
                    if (!announce(tail, 0)) tail = -1;
                }
            }
            for (int e = 0; e < 2 && live; ++e) {
                const int tile = e ? head : tail;
                if (tile < 0) continue;
                const int parts = parts_of(tile), mine = e ? -1 : b - tile * a.n_steps / a.per_cta;
                const int m0 = ((tile + base_tile) % a.m_tiles) * a.mp, m_count = min(a.mp, M - m0), n = row_of(tile);
                for (int c0 = 16 * turn; c0 < m_count; c0 += 16 * kTurns) {
                    uint32_t v[16];
                    float y[16];
#pragma unroll
                    for (int i = 0; i < 16; ++i) y[i] = 0.f;
                    tmem_ld16(v, acc + (uint32_t)c0);
                    tmem_ld_wait(v);
                    for (int q = 0; q < parts; ++q) {
                        const float* part = a.g.partials + ((size_t)q * M + m0 + c0) * n_pad + n;
#pragma unroll
                        for (int i = 0; i < 16; ++i)
                            y[i] += q == mine ? __uint_as_float(v[i]) : c0 + i < m_count && n < N ? __ldcg(part + (size_t)i * n_pad) : 0.f;
                    }
#pragma unroll
                    for (int i = 0; i < 16; ++i) v[i] = __float_as_uint(y[i]);
                    if (n < N) put16(m0 + c0, n, m_count - c0, v);
                }
                __syncwarp();
                if (lane == 0) *ticket_of(tile) = 0;               // zero again for the next call
            }
        }
    }
    if constexpr (CLUSTER) {
        // Each CTA of the cluster adds up its share of the tile's tokens, in ascending k order: the others' parts come into its shared
        // memory as [rank][token][256 rows].  (Written there, not read from there: 4096 x 4096, q = 2, M = 64 13.0 -> 11.3 us.)
        const int tile = b / a.split, rank = b - tile * a.split, share = (a.mp + a.split - 1) / a.split;
        uint8_t* parts = smem + a.exchange;
        __syncwarp();
        if (a.exchange != 0) cluster_wait();                   // every CTA is there
        else cluster_barrier();                                // ... and has read its weights and activations
        if (warp >= kCtrlWarps && have_part) {
            const int blk = ((warp - kCtrlWarps) >> 2) & 1, turn = (warp - kCtrlWarps) >> 3, quad = warp & 3;
            const uint32_t mine = smem_addr(parts) + (uint32_t)((rank * share * kTileRowsN + blk * kBlockRows + quad * 32 + lane) * 4);
            for (int c0 = 16 * turn; c0 < a.mp; c0 += 16 * kTurns) {
                uint32_t v[16];
                tmem_ld16(v, tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)(blk * a.mp + c0));
                tmem_ld_wait(v);
                int owner = c0 / share, token = c0 - owner * share;
#pragma unroll
                for (int i = 0; i < 16; ++i) {
                    if (owner == rank) reinterpret_cast<uint32_t*>(parts)[(mine - smem_addr(parts)) / 4 + token * kTileRowsN] = v[i];
                    else st_cluster_u32(mine + (uint32_t)(token * kTileRowsN * 4), (uint32_t)owner, v[i]);
                    if (++token == share) { token = 0; ++owner; }
                }
            }
        }
        __syncwarp();
        cluster_barrier();                                     // the parts are there
        const int m0 = ((tile + base_tile) % a.m_tiles) * a.mp + rank * share, count = min(min(share, a.mp - rank * share), a.g.M - m0);
        const int row = (tid & 63) * 4, n = ((tile + base_tile) / a.m_tiles) * kTileRowsN + row;
        if (warp >= kCtrlWarps && t1 > t0 && n < a.g.N) {
            grid_dependency_wait();
            const bool plain = !(a.g.flags & (ELUTQ_FLAG_OUT_F32 | ELUTQ_FLAG_ACCUMULATE)) && a.g.N % 4 == 0;
            for (int m = (tid - 32 * kCtrlWarps) / 64; m < count; m += 4 * kBlocks * kTurns * 32 / 64) {
                float4 y = make_float4(0.f, 0.f, 0.f, 0.f);
                for (int q = 0; q < a.split; ++q) {
                    const float4 v = *reinterpret_cast<const float4*>(parts + ((q * share + m) * kTileRowsN + row) * 4);
                    y.x += v.x;
                    y.y += v.y;
                    y.z += v.z;
                    y.w += v.w;
                }
                const size_t at = (size_t)(m0 + m) * a.g.N + n;
                if (plain) {
                    const __half2 lo = __floats2half2_rn(y.x, y.y), hi = __floats2half2_rn(y.z, y.w);
                    *reinterpret_cast<uint2*>(reinterpret_cast<__half*>(a.g.Y) + at) =
                        make_uint2(*reinterpret_cast<const uint32_t*>(&lo), *reinterpret_cast<const uint32_t*>(&hi));
                } else {
                    const float t[4] = {y.x, y.y, y.z, y.w};
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        if (n + i < a.g.N) store_out(a.g, at + i, t[i]);
                }
            }
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 1) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" :: "r"(tmem), "n"(kTmemCols) : "memory");
}

// Tiles that several CTAs share: the parts in ascending k order.  A block per CTA boundary and 8 tokens; the first boundary
// inside a tile stands for the tile.
__global__ void __launch_bounds__(256) hlq_tmem_finalize_kernel(const TmemArgs a) {
    grid_launch_dependents();
    grid_dependency_wait();
    if (a.g.counters != nullptr && __ldcg(a.g.counters) != 0u) return;      // the main kernel refused the blob or gave up
    const int tile = (int)(blockIdx.x + 1) * a.per_cta / a.n_steps;
    const int first = tile * a.n_steps / a.per_cta, parts = (tile * a.n_steps + a.n_steps - 1) / a.per_cta - first + 1;
    if (first != (int)blockIdx.x || parts == 1) return;
    const int n = (tile / a.m_tiles) * kTileRowsN + threadIdx.x, mt0 = (tile % a.m_tiles) * a.mp;
    const int m0 = mt0 + blockIdx.y * 8, m_end = min(mt0 + a.mp, a.g.M);
    if (n >= a.g.N || m0 >= m_end) return;
    const size_t n_pad = (size_t)a.g.n_rb * kTileRows;
    float acc[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) acc[i] = 0.f;
    for (int p = 0; p < parts; p += 4) {
        float v[4][8];
#pragma unroll
        for (int e = 0; e < 4; ++e)
#pragma unroll
            for (int i = 0; i < 8; ++i)
                v[e][i] = (p + e < parts && m0 + i < m_end) ? __ldcg(a.g.partials + ((size_t)(p + e) * a.g.M + m0 + i) * n_pad + n) : 0.f;
#pragma unroll
        for (int e = 0; e < 4; ++e)
#pragma unroll
            for (int i = 0; i < 8; ++i) acc[i] += v[e][i];
    }
#pragma unroll
    for (int i = 0; i < 8; ++i)
        if (m0 + i < m_end) store_out(a.g, (size_t)(m0 + i) * a.g.N + n, acc[i]);
}

using EncodeFn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                              const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                              CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeFn encode_fn() {
    static const EncodeFn fn = [] {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult r;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &r) != cudaSuccess ||
            r != cudaDriverEntryPointSuccess)
            p = nullptr;
        return reinterpret_cast<EncodeFn>(p);
    }();
    return fn;
}

// How the steps of a call are dealt to the SMs: equal shares of all steps, which leaves tiles to be added up from parts; whole tiles,
// which leaves SMs idle; or each tile's K over a cluster of CTAs, which add up through their shared memory.  In us: a step takes
// c when the other SMs do not fight for the L2, 10 % more when all do, the parts 5 (a second kernel 8) and their fp32 bytes at 2.2 TB/s, a cluster's
// sums 1 and 0.035 a token.
// (Measured, equal shares against whole tiles: 28672 x 4096, q = 2, 112 tiles, M = 32: 27 and 25, M = 128: 45 and 32; 57344 x 8192, q = 4,
// 224 tiles, M = 64, the same layer again and again: 127 and 157; 4096 x 14336, q = 3, M = 768, 96 tiles: 99 and 117, M = 1024, 128 tiles: 127 and 120.  Equal
// shares against clusters: 4096 x 4096, q = 2, M = 16 / 64 / 384 11.0 / 14.4 / 31 and 9.3 / 11.3 / 21; 6144 x 4096, q = 4, M = 128 28.5 and
// 19.8; 4096 x 14336, q = 3, M = 64 28.2 and 24.3.)
double step_us(int q, int mp) { return 0.25 + 0.2 * q + 0.0016 * mp; }
// Up to 32 tokens the SMs hardly fight for the L2: equal shares cost whole tiles' steps and 4.4 us with the parts' bytes.  (us, whole tiles / equal shares: 28672 x
// 4096, q = 2, 3, 4, M = 16 23.2, 29.9, 38.3 / 24.2, 29.4, 35.7, M = 32 24.6, 30.8, 40.0 / 26.4, 31.4, 38.6; 28672 x 8192, q = 2, M = 32 46.4 / 41.8.  In two
// rounds, with whole rounds and the rest by clusters third: 43008 x 4096, M = 16, q = 2, 3, 4 43.3, 56.7, 73.1 / 32.1, 39.7, 49.2 / 33.1, 41.2, 52.1; 49382 x 9344, q = 2,
// M = 24 98.9 / 71.3 / 89.0; 45064 x 1024, q = 3, M = 32 18.7 / 18.0 / 19.2; 96638 x 4608, q = 4, M = 16 122.7 / 110.5 / 110.5; 65641 x 1664, q = 1, M = 24 18.3 / 21.9 / 18.3.
// Over 230 calls of 75 to 390 tiles the choice is 0.3 % behind the best of the three, at most 11 % where K is short: 45985 x 1536, q = 2, M = 9 18.9 / 17.1.)
double few_step_us(int q, int mp) { return (q == 1 ? 0.5 : 0.075 + 0.235 * q) + 0.0016 * mp; }
struct Plan { int per_cta, split; double cost; };
Plan plan_of(int q, int mp, int tiles, int n_steps, int num_sms, const int (&max_clusters)[kMaxSplit + 1]) {
    const double c = step_us(q, mp);
    const int steps = tiles * n_steps, whole = (tiles + num_sms - 1) / num_sms * n_steps;
    int share = (steps + num_sms - 1) / num_sms;
    if (share < 2) share = 2;                                 // the partial buffer holds 2 * n_kc slices
    const double ctas = (double)steps / share;
    Plan best = {whole, 1, c * whole};
    const double shared = 1.1 * c * share + (2 * share >= n_steps ? 5.0 : 8.0) + ctas * kTileRowsN * mp * 4.0 / 2.2e6;
    if (shared < best.cost) best = {share, 1, shared};
    for (int s = 2; s <= kMaxSplit && s <= n_steps; ++s) {
        if (max_clusters[s] < tiles) continue;
        const double t = 1.1 * c * ((n_steps + s - 1) / s) + 1.0 + 0.035 * mp;
        if (t < best.cost) best = {n_steps, s, t};
    }
    if (mp <= 32 && best.split == 1 && 2 * share >= n_steps) {
        const double f = few_step_us(q, mp), equal = f * share + 4.4 + ctas * kTileRowsN * mp * 4.0 / 2.2e6;
        best = equal < f * whole ? Plan{share, 1, equal} : Plan{whole, 1, f * whole};
    }
    return best;
}

// What a call is launched as: all tiles by one plan, or whole rounds of whole tiles and the rest of them in a second launch, where that leaves
// less idle (28672 x 4096, q = 2, M = 384, 336 tiles = two rounds and 40 tiles by clusters of three: 93 -> 85 us; M = 320 83 -> 78).
struct Schedule {
    int m_tiles, mp, tiles, n_steps, full;                    // full: tiles of the first launch (all: no second one)
    Plan first, rest;
};
Schedule schedule_of(int q, int M, int N, int K, int num_sms, const int (&max_clusters)[kMaxSplit + 1]) {
    Schedule s;
    s.m_tiles = (M + kMaxTokens - 1) / kMaxTokens;
    s.mp = ((M + s.m_tiles - 1) / s.m_tiles + 15) / 16 * 16;
    s.n_steps = K / 128;
    s.tiles = s.full = (N + kTileRowsN - 1) / kTileRowsN * s.m_tiles;
    s.first = plan_of(q, s.mp, s.tiles, s.n_steps, num_sms, max_clusters);
    s.rest = s.first;
    const int full = s.tiles / num_sms * num_sms;
    if (full > 0 && full < s.tiles) {
        const Plan rounds = {full / num_sms * s.n_steps, 1, (s.mp <= 32 ? few_step_us(q, s.mp) : step_us(q, s.mp)) * (full / num_sms * s.n_steps)};
        const Plan rest = plan_of(q, s.mp, s.tiles - full, s.n_steps, num_sms, max_clusters);
        if (rest.split > 1 && rounds.cost + 6.0 + rest.cost < s.first.cost) {
            s.full = full;
            s.first = rounds;
            s.rest = rest;
        }
    }
    return s;
}

// Clusters of each size that are resident together on the current device (on one that cannot say: GPCs of 18 and 20 SMs).
const int (&cluster_table())[kMaxSplit + 1];

template <int Q>
int launch_tmem_q(const GemmArgs& g, int num_sms, cudaStream_t stream) {
    using C = TmCfg<Q>;
    static bool configured[64] = {};
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev < 0 || dev >= 64) return (int)cudaErrorNotSupported;
    if (!configured[dev]) {
        cudaError_t e = cudaSuccess;
        for (auto kernel : {hlq_tmem_kernel<Q, false, 0>, hlq_tmem_kernel<Q, true, 0>, hlq_tmem_kernel<Q, false, 16>, hlq_tmem_kernel<Q, true, 16>,
                            hlq_tmem_kernel<Q, false, 32>, hlq_tmem_kernel<Q, true, 32>})
            if (e == cudaSuccess) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem);
        if (e != cudaSuccess) return (int)e;
        configured[dev] = true;
    }
    if (!tmem_takes(g.M, g.N, g.K)) return (int)cudaErrorNotSupported;
    const Schedule sch = schedule_of(Q, g.M, g.N, g.K, num_sms, cluster_table());
    TmemArgs a;
    a.g = g;
    a.m_tiles = sch.m_tiles;
    a.mp = sch.mp;
    a.n_steps = sch.n_steps;
    a.ss = (kTmemCols - kBlocks * a.mp) / (kBlocks * kSlotCols);
    if (a.ss > kMaxSlots) a.ss = kMaxSlots;
    const int x_bytes = a.mp * 256, w_bytes = kBlocks * C::UNIT_BYTES;
    auto rings = [&](int room) {                              // two weight chunks at least, four where that leaves four activation steps
        a.ws = 2;
        a.xs = (room - a.ws * w_bytes) / x_bytes;
        while (a.ws < kMaxW && (room - (a.ws + 1) * w_bytes) / x_bytes >= 4) {
            ++a.ws;
            a.xs = (room - a.ws * w_bytes) / x_bytes;
        }
        if (a.xs > kMaxX) a.xs = kMaxX;
    };

    EncodeFn enc = encode_fn();
    if (!enc) return (int)cudaErrorNotSupported;
    CUtensorMap map;
    const cuuint64_t dims[2] = {(cuuint64_t)g.K, (cuuint64_t)g.M}, strides[1] = {(cuuint64_t)g.K * 2};
    const cuuint32_t box[2] = {64, (cuuint32_t)a.mp}, elem[2] = {1, 1};
    if (enc(&map, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, const_cast<__half*>(g.X), dims, strides, box, elem,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
        return (int)cudaErrorInvalidValue;

    auto launch = [&](int tile0, int n_tiles, const Plan& plan) -> int {
        a.tile0 = tile0;
        a.steps = n_tiles * a.n_steps;
        a.per_cta = plan.per_cta;
        a.split = plan.split;
        // A cluster's parts have a place of their own where the rings stay long enough beside it: a CTA need not wait for the others before
        // it writes to them (4096 x 4096, q = 2, M = 16 9.0 -> 8.55 us, M = 32 9.6 -> 9.1, M = 64 11.1 -> 10.4).
        const int parts = a.split > 1 ? a.split * ((a.mp + a.split - 1) / a.split) * kTileRowsN * 4 : 0;
        const bool own = parts > 0 && (kMaxSmem - 1024 - kFixed - 2 * w_bytes - parts) / x_bytes >= 3;
        rings(kMaxSmem - kFixed - (own ? parts + 1024 : 0));
        a.exchange = own ? (a.xs * x_bytes + a.ws * w_bytes + kFixed + 1023) / 1024 * 1024 : 0;
        const int grid = (a.steps + a.per_cta - 1) / a.per_cta * a.split;
        a.reduce = a.per_cta % a.n_steps != 0 && 2 * a.per_cta >= a.n_steps && grid <= kTmemTickets / (4 * kBlocks * kTurns);      // up to three parts
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)grid);
        cfg.blockDim = dim3(kTmThreads);
        cfg.dynamicSmemBytes = own ? a.exchange + parts : a.xs * x_bytes + a.ws * w_bytes + kFixed;
        cfg.stream = stream;
        cudaLaunchAttribute attr[2];
        attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[0].val.programmaticStreamSerializationAllowed = 1;
        attr[1].id = cudaLaunchAttributeClusterDimension;
        attr[1].val.clusterDim.x = (unsigned)a.split;
        attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = a.split > 1 ? 2 : 1;
        // PERM is ahead where the rebuild is the bound and two warps put the activations in order in time and beside the rebuild.  us without and with it, weights
        // from HBM, q = 1, 2, 3, 4: M = 16, 4096 x 4096 7.7, 8.6, 9.7, 11.1 / 7.4, 8.2, 9.3, 10.8; 4096 x 14336 14.6, 18.1, 22.6, 26.6 / 14.2, 16.9, 21.0, 25.7; 28672 x 4096
        // 19.9, 24.9, 31.4, 37.8 / 19.2, 23.3, 29.7, 36.2; 57344 x 8192 59.9, 74.6, 97.3, 123.4 / 56.3, 69.6, 90.5, 116.4.  M = 32 8.2, 9.1, 10.3, 11.6 / 8.1, 9.0, 10.1, 11.3; 15.2, 18.7,
        // 23.2, 27.2 / 14.9, 17.8, 22.0, 25.6; 20.5, 25.3, 32.8, 38.9 / 21.4, 24.8, 31.2, 38.5; 61.6, 76.1, 98.4, 124.9 / 58.7, 72.7, 92.8, 120.6.  Over 264 calls of 40 to 222 tiles and
        // 256 to 8192 k 3 % ahead in the mean; behind at M = 32 with q = 1 and whole tiles (4 % at 28672 x 4096) and with q = 4 and two to six steps (1 to 3 %), where its
        // results are still the more exact ones.  M = 48, two turns of loads a step, 28672 x 4096 25.7, 33.9, 41.4 / 30.0, 34.9, 42.3.  On less than
        // half of the SMs the next kernel's CTAs rebuild meanwhile, the activations' way is what counts: 1000 x 4096, M = 16, q = 2, 3, 4 5.0, 5.2, 5.35 / 5.1, 5.4, 5.55.
        const int perm = 2 * grid <= num_sms || a.mp > 32 ? 0 : a.mp;
        auto kernel = a.split > 1 ? (perm == 16 ? hlq_tmem_kernel<Q, true, 16> : perm == 32 ? hlq_tmem_kernel<Q, true, 32> : hlq_tmem_kernel<Q, true, 0>)
                                  : (perm == 16 ? hlq_tmem_kernel<Q, false, 16> : perm == 32 ? hlq_tmem_kernel<Q, false, 32> : hlq_tmem_kernel<Q, false, 0>);
        cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, map, a);
        count_launch(1);
        if (e != cudaSuccess || a.reduce || a.per_cta % a.n_steps == 0 || grid == 1) return (int)e;
        cfg.gridDim = dim3((unsigned)(grid - 1), (unsigned)((a.mp + 7) / 8));
        cfg.blockDim = dim3(256);
        cfg.dynamicSmemBytes = 0;
        cfg.numAttrs = 1;
        e = cudaLaunchKernelEx(&cfg, hlq_tmem_finalize_kernel, a);
        count_launch(1);
        return (int)e;
    };
    const int ce = launch(0, sch.full, sch.first);
    return ce != 0 || sch.full == sch.tiles ? ce : launch(sch.full, sch.tiles - sch.full, sch.rest);
}

const int (&cluster_table())[kMaxSplit + 1] {
    struct Table { int n[kMaxSplit + 1]; };
    static const Table fallback = {{0, 148, 74, 48, 34, 26, 24, 16, 16}};
    static Table tables[64];
    static std::once_flag once[64];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) {
        (void)cudaGetLastError();
        return fallback.n;
    }
    std::call_once(once[dev], [dev] {
        tables[dev] = fallback;
        if (cudaFuncSetAttribute(hlq_tmem_kernel<4, true, 0>, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem) != cudaSuccess) {
            (void)cudaGetLastError();
            return;
        }
        for (int n = 2; n <= kMaxSplit; ++n) {
            cudaLaunchConfig_t cfg = {};
            cfg.gridDim = dim3((unsigned)(n * 148));
            cfg.blockDim = dim3(kTmThreads);
            cfg.dynamicSmemBytes = kMaxSmem;
            cudaLaunchAttribute attr[1];
            attr[0].id = cudaLaunchAttributeClusterDimension;
            attr[0].val.clusterDim.x = (unsigned)n;
            attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
            cfg.attrs = attr;
            cfg.numAttrs = 1;
            if (cudaOccupancyMaxActiveClusters(&tables[dev].n[n], hlq_tmem_kernel<4, true, 0>, &cfg) != cudaSuccess) {
                tables[dev].n[n] = 0;
                (void)cudaGetLastError();
            }
        }
    });
    return tables[dev].n;
}

}  // namespace

int resident_clusters(int size) { return cluster_table()[size]; }

bool tmem_takes(int M, int N, int K) {
    return (((long long)N + kTileRowsN - 1) / kTileRowsN) * ((M + kMaxTokens - 1) / kMaxTokens) * (K / 128) < (1LL << 30);
}

// Time of a call with more than 128 tokens, fitted to 2300 calls (256 to 57344 rows, K 1024 to 16384, 129 to 2048 tokens; 4 to 6 % off in the
// mean, 9 % for clusters).  plan_of's costs choose between plans; between kernels their constants are not good enough.
double tmem_us(int M, int N, int K, int q, int num_sms) {
    static const double whole_step[5] = {0, 0.22, 0.32, 0.68, 0.96}, whole_tokens[5] = {0, 0.0049, 0.0046, 0.0029, 0.0026};
    static const double share_step[5] = {0, 0.2, 0.3, 0.65, 0.8}, share_tokens[5] = {0, 0.0054, 0.0055, 0.004, 0.0047};
    const Schedule s = schedule_of(q, M, N, K, num_sms, cluster_table());
    const double round = 3.8 + s.n_steps * (whole_step[q] + whole_tokens[q] * s.mp);
    const double rounds = 1.1 + (s.full + num_sms - 1) / num_sms * round;
    if (s.full < s.tiles) return rounds + 5.0 + 0.97 * s.rest.cost;
    if (s.first.split > 1) return 4.1 + s.first.cost * (q == 1 ? 1.1 : 0.97);
    if (s.first.per_cta % s.n_steps == 0) return rounds;
    return 18.0 + s.first.per_cta * (share_step[q] + share_tokens[q] * s.mp);
}

int launch_hlq_tmem(const GemmArgs& g, int q, int num_sms, cudaStream_t stream) {
    switch (q) {
        case 1: return launch_tmem_q<1>(g, num_sms, stream);
        case 2: return launch_tmem_q<2>(g, num_sms, stream);
        case 3: return launch_tmem_q<3>(g, num_sms, stream);
        case 4: return launch_tmem_q<4>(g, num_sms, stream);
        default: return (int)cudaErrorInvalidValue;
    }
}

}  // namespace elutq
