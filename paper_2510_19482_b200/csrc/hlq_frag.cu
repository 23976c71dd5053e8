// Batches of up to ELUTQ_FRAGMENT_MAX_M rows (any at G = 64): bit-planes as MMA fragments, without dequantising.  In two forms, halves and bytes.
//
// Halves: a warp forms the A fragments of mma.sync (16 weight rows x 16 k) in the registers that the MMA reads, with ONE logic
// operation per two weights: of a register with two weight bytes, one in each half, a mask leaves one bit of each half, at
// one of the lowest four bits of the fp16 exponent: 0 or 2^-14, 2^-13, 2^-11, 2^-7.  (The mantissa's bits would do, as
// subnormal numbers, but the tensor core aligns those by their exponent field and loses up to ten bits.)  The activations
// carry the other factor: scaled by 2^c, 2^(c-1), 2^(c-3), 2^(c-7), c such that the largest |x| of the batch row and step
// (128 k) lies just below 2^15.  The scaled values are exact except for elements 2^-22 times smaller than that largest
// one, whose error is at most 2^-33 of it: less than the rounding of the fp32 sums.  So
//
//   Y = sum_g [ sum_j s_j 2^(14-c) D_j + z sum_{k in g} x ],   D_j = the MMAs' sum over the group for plane j,
//
// with the scales applied to the sums in fp32: W_hat is never formed, as in the look-up kernels, and as exact (but next to a value 2^22 times
// larger whose bits are clear).  The MMAs' running sums are truncated, not rounded; a sum runs over one group.
//
//   bytes    Up to four batch rows at G = 128 (BYTES): one logic operation on a word of four weight bytes keeps one bit of each, and what it
//            leaves, 0 or 2^i in every byte, is an operand of the 8-bit integer MMA as it stands: four weights per operation (bits 4-7 as
//            bits 0-3 of the word shifted by 4).  The activations are digits, x_k = 2^(i-F) sum_d 256^d X_d with the X_d the signed bytes of
//            the integer nearest to 2^(F-i) x_k, F such that the largest |x| of the row's step lies just below 2^31.  A value with a bit
//            below that unit 2^(i-F) leaves a rest: the step is contracted a second time, with the rests' digits.  So every activation
//            enters exactly, also next to one that is 2^40 times larger and whose bits are clear.  (Without the second pass, and with i to 7,
//            such sums were off by 2^-23 of the large one.)  There is no rest where the largest |x| is below 15.9, as fp16 has no bit below
//            2^-24, nor of a value that is 2^-17 of the largest or more: 5 of 1000 steps of 4 rows N(0,1) with 1 % of the channels times 20.
//            A group's sums are exact (digits' below 2^16, two of them together below 2^24); a batch row takes four of an MMA's 8
//            columns.  A lane's two digits are put together in its registers, lower and upper ones at the end.
//            Bound: latencies at 20 warps an SM (28672 x 4096, q = 3, M = 4: issue 54 %, logic pipe 44 %, integer MMAs 35 %, LSU 26 %; a warp
//            that does not issue most often finds its math pipe taken or is at the long scoreboard).  us there, q = 2, 3, 4: as halves 25.2, 31.8, 38.7,
//            without the second pass and the shift 23.3, 29.1, 35.6, so 24.1, 29.5, 35.4.
//   k order  an MMA sums over k, so A and B only have to agree on which k a lane holds.  Lane c of a quad takes the bytes of word c
//            of the row's 128 k (bytes: the word as it is, MMA kk the bits 2 kk, 2 kk + 1 of its bytes).  Halves (at G = 64: bytes 2c, 2c+1 of
//            each group): two sub-words with one byte in each half, twice: a left shift by 2 brings the upper copy's bits 0-3 to the four
//            positions, one by 6 the lower copy's bits 4-7 (as multiplications: the logic pipe is the busy one).
//   unit     128 weight rows x 512 k (eight packed tiles, contiguous in the blob: one bulk copy) x 8 NB batch rows (bytes: 2 NB).  The units of
//            a call, output tile by output tile (the batch blocks of a row tile next to each other: its weights come from the L2 again), are
//            dealt to the CTAs (one per SM) in equal contiguous runs, so no SM idles for a wave.  An output tile that several CTAs share
//            is summed in ascending k order (bit-reproducible) by the CTA that finishes it last (a ticket, no CTA waits for another).  Few output
//            tiles are shared by clusters of CTAs instead, whose first CTA adds up.
//   warps    16 compute warps: warp 4 s + r takes step s (128 k) of every unit and rows 32 r .. 32 r + 31 of the tile, so each
//            activation fragment serves two MMAs.  Four activation warps, one per step: scale the unit's activations and
//            lay them out as B fragments, form the group sums; the first of them also loads the weights.
//
// Every wait is bounded; a thread whose wait runs out raises the status word and a CTA-wide flag that ends the other
// warps' waits; copies in flight are waited for (bounded) and the kernel returns.
#include "common.cuh"

namespace elutq {

namespace {

constexpr int kComputeWarps = 16, kComputeThreads = 32 * kComputeWarps;
constexpr int kFragThreads = kComputeThreads + 128;
constexpr int kUnitRows = 128;
constexpr uint32_t kFragWaitLimit = 1u << 22;
constexpr int kMaxRing = 8, kXSlots = 2;        // weight units (at most), units of prepared activations
constexpr int kSumStride = kUnitRows + 4;       // floats per batch row of the sum buffer (conflict-free for fragments)

struct FragArgs {
    GemmArgs g;
    int n_steps;                // 128-k steps of the whole K
    int chunks;                 // units per output tile (512-k chunks)
    int blocks;                 // output tiles per row tile (batch blocks of 8 NB rows; one at G = 128)
    int units, per_cta;         // all units; units of one CTA
    Div by_chunks, by_blocks, by_cta;
    int ws;                     // weight units in flight
    int split;                  // CTAs of a cluster, which share an output tile's chunks (1: no cluster)
    unsigned* tickets;          // zero between calls: one per row tile, or (several blocks) per CTA, for the tile that it begins and does not end
};

enum { kBarWFull = 0, kBarXFull = kBarWFull + kMaxRing, kBarXEmpty = kBarXFull + kXSlots, kNumBars = kBarXEmpty + kXSlots };

template <int Q, int G>
struct FragCfg {
    static constexpr int W = G / 8, NSG = 128 / G;
    static constexpr int PLANE_BYTES = 1024 * Q;
    static constexpr int TILE_BYTES = PLANE_BYTES + 128 * (NSG * (Q + 1));
    static constexpr int UNIT_BYTES = 8 * TILE_BYTES;
};

__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
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
__device__ __forceinline__ bool elect_one() {
    uint32_t e;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(e));
    return e != 0;
}
__device__ __forceinline__ uint32_t lds32(uint32_t addr) {
    uint32_t v;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(addr));
    return v;
}
__device__ __forceinline__ uint32_t lds16(uint32_t addr) {
    unsigned short v;
    asm volatile("ld.shared.u16 %0, [%1];" : "=h"(v) : "r"(addr));
    return v;
}
__device__ __forceinline__ uint4 lds128(uint32_t addr) {
    uint4 v;
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr));
    return v;
}
__device__ __forceinline__ void mma_16816(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
// Weights' bits (unsigned bytes) times digits (signed ones); `first` begins a sum.
__device__ __forceinline__ void mma_16832(int (&c)[4], bool first, uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
    const int z[4] = {first ? 0 : c[0], first ? 0 : c[1], first ? 0 : c[2], first ? 0 : c[3]};
    asm("mma.sync.aligned.m16n8k32.row.col.s32.u8.s8.s32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%10, %11, %12, %13};"
        : "=r"(c[0]), "=r"(c[1]), "=r"(c[2]), "=r"(c[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1), "r"(z[0]), "r"(z[1]), "r"(z[2]), "r"(z[3]));
}
__device__ __forceinline__ float half_bits(uint32_t v) { return __half2float(__ushort_as_half((unsigned short)v)); }

// slot and parity of the n-th use of a ring, advanced without divisions
struct Ring {
    int len, i;
    uint32_t phase;
    __device__ __forceinline__ Ring(int n) : len(n), i(0), phase(0) {}
    __device__ __forceinline__ void next() {
        if (++i == len) { i = 0; phase ^= 1u; }
    }
};

// BYTES: a word per digit of a lane's four elements d (integers, |d| <= 2^31 - 2^23) to its places o, o + 16, ... in the B fragments.
__device__ __forceinline__ void store_digits(uint32_t* o, uint32_t (&d)[4]) {
#pragma unroll
    for (int e = 0; e < 4; ++e) d[e] = (d[e] + 0x00808080u) ^ 0x00808080u;      // balanced, so that the lower three digits are signed bytes too
    const uint32_t lo01 = __byte_perm(d[0], d[1], 0x5140), hi01 = __byte_perm(d[0], d[1], 0x7362);
    const uint32_t lo23 = __byte_perm(d[2], d[3], 0x5140), hi23 = __byte_perm(d[2], d[3], 0x7362);
    o[0] = __byte_perm(lo01, lo23, 0x5410);
    o[16] = __byte_perm(lo01, lo23, 0x7632);
    o[32] = __byte_perm(hi01, hi23, 0x5410);
    o[48] = __byte_perm(hi01, hi23, 0x7632);
}

__device__ __forceinline__ float power_of_two(int e) { return __int_as_float((127 + e) << 23); }

// BYTES: what the digits of a step leave of the batch rows' values: fractions of a unit, which are multiples of 2^-13 (of 2^-24 in the value, whose
// unit is at most 2^(3-14)), times 2^15, in digits.  x: the lane's first element in row 0; meta: the rows' factors 2^-F.
__device__ __noinline__ void store_rest(const unsigned short* x, int K, int M, int rows, int bit, const float* meta, uint32_t* frag) {
#pragma unroll 1
    for (int m = 0; m < rows; ++m) {
        uint32_t d[4] = {};
        if (m < M) {
            const int F = 127 - (int)(__float_as_uint(meta[m]) >> 23);
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const float v = half_bits(__ldg(x + (size_t)m * K + 8 * e)) * power_of_two(F - (bit & 3));
                d[e] = (uint32_t)__float2int_rn((v - rintf(v)) * 32768.f);
            }
        }
        store_digits(frag + (m >> 1) * 256 + (m & 1) * 64, d);
    }
}

// What chunks [chunk, end) add to Y[m][n], element by element (G = 128).  For infinities and NaN, of which digits cannot say what a bit
// leaves: an infinite activation is none where its bit is 0, an infinite scale or offset times sums of both signs is an infinity.  Some 500
// instructions a step; no call with finite values comes here.
template <int Q>
__device__ __noinline__ float plain_sum(const __half* __restrict__ x, const uint8_t* __restrict__ tiles, size_t chunk_bytes, int l, int chunk, int end, int n_steps,
                                        unsigned flags) {
    using C = FragCfg<Q, 128>;
    const int last = min(4 * end, n_steps);
    float y = 0.f;
#pragma unroll 1
    for (int s = 4 * chunk; s < last; ++s) {                  // (x: row m; tiles: the row block's of chunk 0; l: the row in it)
        const int u = (s >> 1) & 1, h = s & 1;
        const uint8_t* tb = tiles + (size_t)(s >> 2) * chunk_bytes;
        const uint8_t* planes = tb + (u * Q * 32 + 16 * h + l) * 16;
        const uint8_t* params = tb + C::PLANE_BYTES + (16 * h + l) * 4;
        const unsigned short* xs = reinterpret_cast<const unsigned short*>(x) + s * 128;
        float sum[Q + 1] = {};                                // of the planes; of the group
#pragma unroll 1
        for (int b = 0; b < 16; ++b) {
#pragma unroll 1
            for (int i = 0; i < 8; ++i) {
                const float v = half_bits(__ldg(xs + 8 * b + i));
#pragma unroll
                for (int j = 0; j < Q; ++j) sum[j] += planes[j * 512 + ((b - l) & 15)] >> i & 1 ? v : 0.f;
                sum[Q] += v;
            }
        }
        float own = 0.f;
#pragma unroll
        for (int j = 0; j <= Q; ++j) {                        // scales, offset
            const int rec = u * (Q + 1) + j;
            const float p = half_bits(*reinterpret_cast<const unsigned short*>(params + (rec >> 1) * 128 + (rec & 1) * 2));
            if (!(flags & (j < Q ? ELUTQ_FLAG_OFFSET_ONLY : ELUTQ_FLAG_SKIP_OFFSET))) own = fmaf(p, sum[j], own);
        }
        y += own;
    }
    return y;
}

// NB = blocks of 8 columns (MMA N): of 8 batch rows, or (BYTES) of two with four digits each.  FOLD: long runs of units, whose sums are
// put by every two units.  SPLIT: the chunks of an output tile are shared by the CTAs of a cluster.
template <int Q, int G, int NB, bool FOLD, bool BYTES, bool SPLIT>
__global__ void __launch_bounds__(kFragThreads, 1) hlq_frag_kernel(const FragArgs a) {
    using C = FragCfg<Q, G>;
    static_assert(G == 128 || G == 64, "");
    constexpr int NSG = C::NSG;                               // groups per step: 1 or 2
    constexpr int MP = (BYTES ? 2 : 8) * NB;
    constexpr bool kStepSum = BYTES || NB == 1;
    static_assert(!(kStepSum && FOLD), "");
    constexpr int XF_BYTES = 8192 * NB;                       // B fragments of a unit: [digits, rest (BYTES)][step][block][2 or 4][lane] 16 bytes
    static_assert(!BYTES || G == 128, "");
    constexpr int XM_STEP = (1 + NSG) * MP + (BYTES ? 1 : 0); // per step: factor and group sums of every batch row (BYTES: whether there is a rest)
    constexpr int XM_FLOATS = 4 * XM_STEP;
    extern __shared__ __align__(1024) uint8_t smem[];
    uint8_t* sX = smem;
    uint8_t* sW = sX + kXSlots * XF_BYTES;
    float* sM = reinterpret_cast<float*>(sW + a.ws * C::UNIT_BYTES);
    float* sSum = sM + kXSlots * XM_FLOATS;                   // [step][MP][kSumStride]
    uint64_t* bars = reinterpret_cast<uint64_t*>(sSum + 4 * MP * kSumStride);
    volatile uint32_t* give_up = reinterpret_cast<uint32_t*>(bars + kNumBars);
    volatile uint32_t* ticket_box = give_up + 1;
    volatile uint32_t* lost_box = ticket_box + 1;             // split: another CTA of the cluster gave up
    float* sParts = reinterpret_cast<float*>(bars + kNumBars + 2);        // split: the other CTAs' sums, [rank - 1][MP][kUnitRows]
    const uint32_t bar0 = smem_addr(bars);
    auto bar = [&](int i) { return bar0 + 8u * (uint32_t)i; };

    const int tid = threadIdx.x, lane = tid & 31;
    const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);   // warp-uniform for the compiler too
    uint4 h0;
    uint2 h1;
    blob_header_load(a.g.tiles, h0, h1);
    if (tid == 0) {
        auto init = [&](int i, int n) { asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" :: "r"(bar(i)), "r"(n) : "memory"); };
        for (int i = 0; i < kMaxRing; ++i) init(kBarWFull + i, 1);
        for (int i = 0; i < kXSlots; ++i) {
            init(kBarXFull + i, 4);
            init(kBarXEmpty + i, kComputeWarps);              // a unit is done with: its activations and its weights
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        *give_up = 0;
        *lost_box = 0;
    }
    __syncthreads();
    if constexpr (SPLIT) cluster_arrive();                        // (the box is clear, the CTA is there: awaited before a peer writes)

    const int b = blockIdx.x, C_ = a.chunks;
    int u0 = b * a.per_cta, u1 = min(a.units, u0 + a.per_cta), rank = 0;
    if constexpr (SPLIT) {                                    // a tile's chunks in ascending shares
        const int tile = b / a.split;
        rank = b - tile * a.split;
        u0 = tile * C_ + C_ * rank / a.split;
        u1 = tile * C_ + C_ * (rank + 1) / a.split;
    }
    const bool refused = !blob_header_ok(h0, h1, Q, G, a.g.N, a.g.K);
    if (refused) {                                            // before any tile is read; the same answer in every thread: no work
        u1 = u0;
        if (tid == 0 && a.g.counters != nullptr) atomicExch(a.g.counters, kStatusBlobMismatch);
    }
    auto row_tile = [&](int tile) { return G == 128 ? tile : a.by_blocks.of(tile); };
    auto batch0 = [&](int tile) { return G == 128 ? 0 : (tile - a.by_blocks.of(tile) * a.blocks) * MP; };
    const uint32_t limit = a.g.wait_limit ? a.g.wait_limit : kFragWaitLimit;
    // Bounded wait; false once this CTA has given up.
    auto wait_many = [&](auto poll) {
        for (uint32_t n = 0; n < limit; ++n) {
            if (poll()) return true;
            if (*give_up) return false;
        }
        *give_up = 1;
        if (a.g.counters != nullptr) atomicExch(a.g.counters, kStatusWaitExpired);
        return false;
    };
    auto steps_of = [&](int chunk) { return min(4, a.n_steps - 4 * chunk); };
    const int gq = lane >> 2, c = lane & 3;                   // fragment row (and batch row of B), position in the quad
    const int M = a.g.M, N = a.g.N;
    grid_launch_dependents();

    if (warp >= kComputeWarps) {
        // ---- activation warps ------------------------------------------------------------------------------------------------
        const int step = warp - kComputeWarps;
        const bool use_offset = !(a.g.flags & ELUTQ_FLAG_SKIP_OFFSET);
        const bool loads = !test_stalls(a.g.flags);           // (test flag: nothing is loaded, the waits run out)
        int wu = u0, wslot = 0;                               // next unit whose weights are to be loaded, its slot
        auto load_weights = [&](int upto) {                   // by one elected lane; slot = unit number in the CTA mod ws
            for (; wu < upto; ++wu) {
                const int tile = a.by_chunks.of(wu), rb0 = row_tile(tile) * 8, slot = wslot;
                const uint32_t bytes = (uint32_t)(min(8, a.g.n_rb - rb0) * C::TILE_BYTES);
                if (elect_one()) {
                    mbar_expect(bar(kBarWFull + slot), bytes);
                    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                                 :: "r"(smem_addr(sW) + (uint32_t)(slot * C::UNIT_BYTES)),
                                    "l"(a.g.tiles + ((size_t)(wu - tile * C_) * a.g.n_rb + rb0) * C::TILE_BYTES), "r"(bytes), "r"(bar(kBarWFull + slot))
                                 : "memory");
                }
                __syncwarp();
                if (++wslot == a.ws) wslot = 0;
            }
        };
        // weights do not depend on the previous kernel: the first units are requested before the dependency wait
        if (step == 0 && loads) load_weights(min(u1, u0 + a.ws));
        grid_dependency_wait();

        // BYTES: the lane's word of a row's plane bytes and bit position, and its place among the B fragments.
        const int bit = lane & 7, word = lane >> 3, place = (bit >> 2) * 128 + word * 4 + (bit & 3);
        uint32_t raw_h[BYTES ? MP : 1][4];
        // The lane's four 16-byte pieces (8 k each) of a batch row and step: the low and the high bytes of the two sub-words.
        const int piece[2][2] = {{G == 128 ? 4 * c : 2 * c, G == 128 ? 4 * c + 2 : 2 * c + 1},
                                 {G == 128 ? 4 * c + 1 : 8 + 2 * c, G == 128 ? 4 * c + 3 : 8 + 2 * c + 1}};
        uint4 raw[NB][2][2];
        auto fetch = [&](int mb, int chunk) {
            if constexpr (BYTES) {
#pragma unroll
                for (int m = 0; m < MP; ++m)
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const int k = chunk * kChunkK + step * 128 + (4 * word + e) * 8 + bit;
                        raw_h[m][e] = (mb + m < M && k < a.g.K) ? __ldg(reinterpret_cast<const unsigned short*>(a.g.X) + (size_t)(mb + m) * a.g.K + k) : 0u;
                    }
            } else {
#pragma unroll
            for (int nb = 0; nb < NB; ++nb)
#pragma unroll
                for (int q = 0; q < 2; ++q)
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        const int m = mb + 8 * nb + gq, k = chunk * kChunkK + step * 128 + piece[q][e] * 8;
                        raw[nb][q][e] = (m < M && k < a.g.K) ? __ldg(reinterpret_cast<const uint4*>(a.g.X + (size_t)m * a.g.K + k)) : make_uint4(0, 0, 0, 0);
                    }
            }
        };
        int tile = a.by_chunks.of(u0), chunk = u0 - tile * C_, mb = batch0(tile);
        if (u0 < u1) fetch(mb, chunk);
        for (int u = u0; u < u1; ++u) {
            const int t = u - u0, slot = t & 1;
            if (!__all_sync(0xffffffffu, wait_many([&]() { return mbar_try(bar(kBarXEmpty + slot), (uint32_t)((t >> 1) & 1) ^ 1u); }))) break;
            if (step == 0 && t >= 2 && loads) load_weights(min(u1, u - 2 + a.ws + 1));      // the unit two back has been read
            if constexpr (BYTES) {
                const int k0 = chunk * kChunkK + step * 128;
                float x[MP][4];
                uint32_t top[MP];
#pragma unroll
                for (int m = 0; m < MP; ++m) {
                    top[m] = __reduce_max_sync(0xffffffffu, max(max(raw_h[m][0] & 0x7fffu, raw_h[m][1] & 0x7fffu), max(raw_h[m][2] & 0x7fffu, raw_h[m][3] & 0x7fffu)));
#pragma unroll
                    for (int e = 0; e < 4; ++e) x[m][e] = half_bits(raw_h[m][e]);
                }
                const bool there = step < steps_of(chunk);
                if (++chunk == C_) {
                    chunk = 0;
                    mb = batch0(++tile);
                }
                if (u + 1 < u1) fetch(mb, chunk);             // (in flight while this unit's are worked on)
                if (there) {
                    uint32_t* frag = reinterpret_cast<uint32_t*>(sX + slot * XF_BYTES) + step * (NB * 256) + place;
                    float* meta = sM + slot * XM_FLOATS + step * XM_STEP;
                    bool rest = false;
                    float four[MP];
#pragma unroll
                    for (int m = 0; m < MP; ++m) {
                        const int F = 45 - min(max((int)((top[m] + 8u) >> 10), 1), 31);         // |x| 2^F <= 2^31 - 9 2^20
                        const float scale = power_of_two(F - (bit & 3));
                        uint32_t d[4];
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            const int n = __float2int_rn(x[m][e] * scale);
                            rest |= (float)n != x[m][e] * scale;
                            d[e] = (uint32_t)n;
                        }
                        store_digits(frag + (m >> 1) * 256 + (m & 1) * 64, d);
                        four[m] = (x[m][0] + x[m][1]) + (x[m][2] + x[m][3]);
                        // (a row that is not all finite: the write-out sums it anew)
                        if (lane == 0) meta[m] = top[m] < 0x7c00u ? power_of_two(-F) : __int_as_float(0x7fffffff);
                    }
                    // the rows' sums over the lanes, row m in lanes m, m + MP, ...
                    auto fold = [&](float even, float odd, int b) {
                        const bool up = (lane & b) != 0;
                        return (up ? odd : even) + __shfl_xor_sync(0xffffffffu, up ? even : odd, b);
                    };
                    float total = fold(four[0], four[1], 1);
                    if constexpr (MP == 4) total = fold(total, fold(four[2], four[3], 1), 2);
#pragma unroll
                    for (int o = MP; o < 32; o <<= 1) total += __shfl_xor_sync(0xffffffffu, total, o);
                    if (lane < MP) meta[MP + lane] = total;
                    rest = __any_sync(0xffffffffu, rest);
                    if (lane == 0) reinterpret_cast<uint32_t*>(meta)[2 * MP] = rest ? 1u : 0u;
                    if (__builtin_expect(rest, 0)) {
                        __syncwarp();
                        store_rest(reinterpret_cast<const unsigned short*>(a.g.X) + k0 + 32 * word + bit, a.g.K, M, MP, bit, meta, frag + NB * 1024);
                    }
                }
            }
            if (!BYTES && step < steps_of(chunk)) {
                uint4* frag = reinterpret_cast<uint4*>(sX + slot * XF_BYTES) + step * (NB * 128) + lane;
                float* meta = sM + slot * XM_FLOATS + step * XM_STEP;
#pragma unroll
                for (int nb = 0; nb < NB; ++nb) {
                    __half2 v[2][2][4];
#pragma unroll
                    for (int q = 0; q < 2; ++q)
#pragma unroll
                        for (int e = 0; e < 2; ++e) {
                            const uint32_t r[4] = {raw[nb][q][e].x, raw[nb][q][e].y, raw[nb][q][e].z, raw[nb][q][e].w};
#pragma unroll
                            for (int i = 0; i < 4; ++i) v[q][e][i] = *reinterpret_cast<const __half2*>(&r[i]);
                        }
                    // group sums: the batch rows as A rows, times ones; a sub-word's activations belong to one group
                    float sum[2][4] = {};
                    __half2 mx = __habs2(v[0][0][0]);         // largest |x| of the row's step
#pragma unroll
                    for (int q = 0; q < 2; ++q)
#pragma unroll
                        for (int e = 0; e < 2; ++e)
#pragma unroll
                            for (int i = 0; i < 4; i += 2) {
                                mma_16816(sum[q], *reinterpret_cast<const uint32_t*>(&v[q][e][i]), 0u,
                                          *reinterpret_cast<const uint32_t*>(&v[q][e][i + 1]), 0u, 0x3c003c00u, 0x3c003c00u);
                                mx = __hmax2(mx, __hmax2(__habs2(v[q][e][i]), __habs2(v[q][e][i + 1])));
                            }
                    uint32_t top = __half_as_ushort(__hmax(__low2half(mx), __high2half(mx)));
                    top = max(top, __shfl_xor_sync(0xffffffffu, top, 1));
                    top = max(top, __shfl_xor_sync(0xffffffffu, top, 2));
                    const int ex = max(1, (int)(top >> 10)), cx = 29 - ex, c1 = min(cx, 14);      // x 2^cx < 2^15
                    const bool infinite = top == 0x7c00u && use_offset;
                    if (c == 0) {
                        meta[8 * nb + gq] = __uint_as_float(infinite ? 0x7f000000u : (uint32_t)(127 + 14 - cx) << 23);
                        if (NSG == 1) {
                            meta[MP + 8 * nb + gq] = sum[0][0] + sum[1][0];
                        } else {
                            meta[MP + 8 * nb + gq] = sum[0][0];
                            meta[2 * MP + 8 * nb + gq] = sum[1][0];
                        }
                    }
                    // x 2^c1 exactly, then 2^(cx - c1) and what the bit's mask leaves to do (2^cx may exceed fp16)
                    const uint32_t f1b = (uint32_t)(15 + c1) * 0x04000400u, f2b = (uint32_t)(15 + cx - c1) * 0x04000400u;
                    const __half2 f1 = *reinterpret_cast<const __half2*>(&f1b);
#pragma unroll
                    for (int q = 0; q < 2; ++q) {
                        uint32_t o[8];
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            const __half2 lo = __hmul2(v[q][0][i], f1), hi = __hmul2(v[q][1][i], f1);
                            const uint32_t l = *reinterpret_cast<const uint32_t*>(&lo), h = *reinterpret_cast<const uint32_t*>(&hi);
                            const uint32_t pr[2] = {__byte_perm(l, h, 0x5410), __byte_perm(l, h, 0x7632)};
#pragma unroll
                            for (int e = 0; e < 2; ++e) {
                                constexpr uint32_t kDown[4] = {0u, 1u, 3u, 7u};
                                const uint32_t fb = f2b - kDown[(2 * i + e) & 3] * 0x04000400u;
                                const __half2 r = __hmul2(*reinterpret_cast<const __half2*>(&pr[e]), *reinterpret_cast<const __half2*>(&fb));
                                o[2 * i + e] = *reinterpret_cast<const uint32_t*>(&r);
                            }
                        }
                        frag[(nb * 4 + 2 * q) * 32] = make_uint4(o[0], o[1], o[2], o[3]);
                        frag[(nb * 4 + 2 * q + 1) * 32] = make_uint4(o[4], o[5], o[6], o[7]);
                    }
                    // An infinity: with the offset term the row's results are not finite whatever its other activations are.  As an
                    // operand it would make 0 * infinity = NaN of every bit that is not set.  2^15 in its place (less what the bit's mask
                    // does), zeros elsewhere and a factor of 2^127 make an infinity of the set bits' sum, and 0 of none.
                    if (infinite) {
                        uint32_t* w = reinterpret_cast<uint32_t*>(frag + nb * 128);
#pragma unroll 1
                        for (int i = 0; i < 16; ++i) {
                            const uint32_t r = w[(i >> 2) * 128 + (i & 3)], size = r & 0x7fff7fffu;
                            const uint32_t inf = __vcmpeq2(size, 0x7c007c00u), nan = __vcmpgtu2(size, 0x7c007c00u);
                            const uint32_t in_place = 0x78007800u - (0x7310u >> (4 * (i & 3)) & 15u) * 0x04000400u;
                            w[(i >> 2) * 128 + (i & 3)] = (inf & ((r & 0x80008000u) | in_place)) | (nan & r);
                        }
                    }
                }
            }
            if constexpr (!BYTES) {
                if (++chunk == C_) {
                    chunk = 0;
                    mb = batch0(++tile);
                }
                if (u + 1 < u1) fetch(mb, chunk);
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(bar(kBarXFull + slot));
        }
        if (step == 0)                                        // copies in flight land before the CTA may leave (given up or not)
            for (int n = max(u0, wu - a.ws); n < wu; ++n)
                for (uint32_t t = 0; t < kFragWaitLimit && !mbar_try(bar(kBarWFull + (n - u0) % a.ws), (uint32_t)((n - u0) / a.ws) & 1u); ++t) {}
        if constexpr (SPLIT) {
            __syncwarp();
            cluster_wait();
            cluster_arrive();
            cluster_wait();
        }
        __syncthreads();
        return;
    }

    // ---- compute warps -------------------------------------------------------------------------------------------------------
    const int step = warp >> 2, rp = warp & 3;                // the warp's 128 k of every chunk, its 32 rows of the tile
    const bool use_planes = !(a.g.flags & ELUTQ_FLAG_OFFSET_ONLY), use_offset = !(a.g.flags & ELUTQ_FLAG_SKIP_OFFSET);
    const uint32_t offset_mask = use_offset ? 0xffffffffu : 0u;
    const bool add_offset = use_offset && !(lane & 1);        // BYTES: by the lanes of the lower digits

    // Where the lane finds its bytes of rows gq and gq + 8 of a packed tile (the layout rotates groups and bytes by the row):
    // two 32-bit words at off0 / off1 (G = 64: per group), of which the selectors pick the bytes of a sub-word.
    uint32_t off0[2], off1[2], sel[2];
#pragma unroll
    for (int e = 0; e < 2; ++e) {
        const int l = gq + 8 * e;
        const uint32_t vec = (uint32_t)((2 * rp) * C::TILE_BYTES + ((step >> 1) * Q * 32 + 16 * (step & 1) + l) * 16);
        const int ii = G == 128 ? (4 * c - l) & 15 : (2 * c - l) & 7;
        off0[e] = vec + (uint32_t)(ii & ~3);
        off1[e] = vec + (uint32_t)(((ii & ~3) + 4) & (C::W - 1));
    }
    {   // a sub-word's low byte goes to bytes 0 and 1, its high byte to bytes 2 and 3
        const uint32_t s = (uint32_t)((G == 128 ? 4 * c - gq : 2 * c - gq) & 3);
        sel[0] = s * 0x0011u + (s + (G == 128 ? 2u : 1u)) * 0x1100u;
        sel[1] = G == 128 ? sel[0] + 0x1111u : sel[0];
    }
    const int word_shift = 8 * ((0 - gq) & 3);                // BYTES: the lane's word begins there
    uint32_t by4 = 4u, by64 = 64u;                            // opaque, so that the products stay products
    asm volatile("" : "+r"(by4), "+r"(by64));
    const uint32_t poff = (uint32_t)((2 * rp) * C::TILE_BYTES + C::PLANE_BYTES + (16 * (step & 1) + gq) * 4);
    // fp16 bits of component `comp` of the group at position p, row r (gq + 8 r of the warp's 32); tb = the unit's weights
    auto parameter = [&](uint32_t tb, int r, int p, int comp) {
        const int v = NSG == 1 ? 0 : (p - (r & 1)) & 1;       // (rows gq + 8 start with the other group)
        const int rec = ((step >> 1) * NSG + v) * (Q + 1) + comp;
        return lds16(tb + poff + (uint32_t)((r >> 1) * C::TILE_BYTES + (r & 1) * 32 + (rec >> 1) * 128 + (rec & 1) * 2));
    };

    grid_dependency_wait();
    const size_t n_pad = (size_t)a.g.n_rb * kTileRows;
    const bool plain = !(a.g.flags & (ELUTQ_FLAG_OUT_F32 | ELUTQ_FLAG_ACCUMULATE));
    auto put = [&](int m, int n, float y) {
        if (plain) reinterpret_cast<__half*>(a.g.Y)[(size_t)m * N + n] = __float2half_rn(y);
        else store_out(a.g, (size_t)m * N + n, y);
    };
    auto compute_sync = []() { asm volatile("bar.sync 1, 512;" ::: "memory"); };
    auto compute_any = [](bool mine) {                        // the same barrier; one answer for all compute threads
        int any;
        asm volatile("{\n\t.reg .pred p, r;\n\tsetp.ne.s32 p, %1, 0;\n\tbar.red.or.pred r, 1, 512, p;\n\tselp.s32 %0, 1, 0, r;\n\t}"
                     : "=r"(any) : "r"((int)mine) : "memory");
        return any != 0;
    };
    // The CTA that came last to a shared output tile adds the parts in ascending k order (all compute threads call this), four at a time in pairs:
    // fewer roundings than in one chain, in the same time (error of the fp32 result, chain / pairs, q = 4: 1024 x 14336, M = 8 1.1e-7 / 1.0e-7,
    // M = 4 8.0e-8 / 6.8e-8, G = 64 1.1e-7 / 1.0e-7; 256 x 65536, M = 8 1.9e-7 / 1.3e-7; the look-up kernel there 1.1e-7, 7.6e-8, 1.1e-7, 1.5e-7).
    auto parts_of = [&](int tile) { return a.by_cta.of(tile * C_ + C_ - 1) - a.by_cta.of(tile * C_) + 1; };
    auto ticket_of = [&](int tile) { return a.tickets + (G == 128 || a.blocks == 1 ? tile : a.by_cta.of(tile * C_)); };
    auto finish_tile = [&](int tile) {
        if (tile < 0 || *ticket_box == 0u) return;
        const int n = row_tile(tile) * kUnitRows + (tid & (kUnitRows - 1)), mb = batch0(tile), me = min(M, mb + MP);
        const int parts = parts_of(tile);
        if (n >= N) return;
        const float* p0 = a.g.partials + n;
        for (int m0 = mb + (tid >> 7); m0 < me; m0 += 16) {
            float y[4] = {0.f, 0.f, 0.f, 0.f};
            for (int p = 0; p < parts; p += 4) {
                float v[4][4];
#pragma unroll
                for (int e = 0; e < 4; ++e)
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        v[e][i] = (p + e < parts && m0 + 4 * i < me) ? __ldcg(p0 + ((size_t)(p + e) * M + m0 + 4 * i) * n_pad) : 0.f;
#pragma unroll
                for (int i = 0; i < 4; ++i) y[i] += (v[0][i] + v[1][i]) + (v[2][i] + v[3][i]);       // (pairs: see above)
            }
#pragma unroll
            for (int i = 0; i < 4; ++i)
                if (m0 + 4 * i < me) put(m0 + 4 * i, n, y[i]);
        }
    };

    constexpr int NE = BYTES ? 2 : 4;                         // sums of a lane: rows gq, gq + 8 (times batch rows 2c, 2c + 1)
    float* own_sum = sSum + (step * MP + (BYTES ? c >> 1 : 2 * c)) * kSumStride + 32 * rp + gq;      // where the lane's sums go in the buffer
    auto sum_at = [](int nb, int t, int i) { return BYTES ? 2 * nb * kSumStride + 16 * t + 8 * i : (8 * nb + (i & 1)) * kSumStride + 16 * t + 8 * (i >> 1); };

    auto sum_of = [&](int m, int row, int n, int chunk, int end) {         // this CTA's part of Y[mb + m][n]
        float y = sSum[m * kSumStride + row];
#pragma unroll
        for (int s = 1; s < 4; ++s) y += sSum[(s * MP + m) * kSumStride + row];
        if constexpr (BYTES) {
            if (__builtin_expect((__float_as_uint(y) & 0x7f800000u) == 0x7f800000u, 0) && n < N)
                y = plain_sum<Q>(a.g.X + (size_t)m * a.g.K, a.g.tiles + (size_t)(n >> 4) * C::TILE_BYTES, (size_t)a.g.n_rb * C::TILE_BYTES, n & 15, chunk, end,
                                 a.n_steps, a.g.flags);
        }
        return y;
    };

    Ring w(a.ws), x(kXSlots);
    bool live = true, gone = refused;                         // gone: the compute warps gave up together
    int pending = -1;                                         // output tile whose ticket has been taken and not looked at
    for (int u = u0; u < u1 && live;) {
        const int tile = a.by_chunks.of(u), chunk0 = u - tile * C_;
        const int n_units = min(C_ - chunk0, u1 - u);
        u += n_units;
        if (FOLD) compute_sync();                             // the buffer has been read
        float acc[2][NB][NE];
#pragma unroll
        for (int t = 0; t < 2; ++t)
#pragma unroll
            for (int nb = 0; nb < NB; ++nb)
#pragma unroll
                for (int i = 0; i < NE; ++i) acc[t][nb][i] = 0.f;

        for (int cu = 0; cu < n_units; ++cu) {
            live = __all_sync(0xffffffffu, wait_many([&]() {
                return mbar_try(bar(kBarWFull + w.i), w.phase) & mbar_try(bar(kBarXFull + x.i), x.phase);
            }));
            if (!live) break;
            if (BYTES && step < steps_of(chunk0 + cu)) {
                // Lane c of a quad holds two digits of batch row c / 2 of every block: the lower two, or the upper two times 2^16
                const uint8_t* wb = sW + w.i * C::UNIT_BYTES;
                const uint4* xb = reinterpret_cast<const uint4*>(sX + x.i * XF_BYTES) + step * (NB * 64) + lane;
                const float* meta = sM + x.i * XM_FLOATS + step * XM_STEP;
                float own[2][NB][2];
                const uint32_t pb = smem_addr(wb);
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    const float z = half_bits(parameter(pb, r, 0, Q));
#pragma unroll
                    for (int nb = 0; nb < NB; ++nb) own[r >> 1][nb][r & 1] = add_offset ? z * meta[MP + 2 * nb + (c >> 1)] : 0.f;
                }
                if (use_planes) {
                    uint4 xd[NB][2];                          // B fragments, held over the planes
                    float fac[NB];
                    auto load_digits = [&](int pass, float unit) {
#pragma unroll
                        for (int nb = 0; nb < NB; ++nb) {
                            xd[nb][0] = xb[pass * (NB * 256) + nb * 64];
                            xd[nb][1] = xb[pass * (NB * 256) + nb * 64 + 32];
                            fac[nb] = meta[2 * nb + (c >> 1)] * ((c & 1) ? 65536.f * unit : unit);
                        }
                    };
                    auto plane = [&](int j) {
                        uint32_t pw[4];
#pragma unroll
                        for (int r = 0; r < 4; ++r) {
                            const uint8_t* tb = wb + (r >> 1) * C::TILE_BYTES + j * 512;
                            pw[r] = __funnelshift_r(*reinterpret_cast<const uint32_t*>(tb + off0[r & 1]), *reinterpret_cast<const uint32_t*>(tb + off1[r & 1]), word_shift);
                        }
                        int d[2][NB][4];
#pragma unroll
                        for (int kk = 0; kk < 4; ++kk) {      // two bit positions of the words: 32 k of each row
                            uint32_t f[4][2];
#pragma unroll
                            for (int r = 0; r < 4; ++r)
#pragma unroll
                                for (int i = 0; i < 2; ++i) f[r][i] = (kk < 2 ? pw[r] : pw[r] >> 4) & (0x01010101u << (2 * (kk & 1) + i));
#pragma unroll
                            for (int nb = 0; nb < NB; ++nb) {
                                const uint4 xv = xd[nb][kk >> 1];
#pragma unroll
                                for (int t = 0; t < 2; ++t)
                                    mma_16832(d[t][nb], kk == 0, f[2 * t][0], f[2 * t + 1][0], f[2 * t][1], f[2 * t + 1][1], kk & 1 ? xv.z : xv.x,
                                              kk & 1 ? xv.w : xv.y);
                            }
                        }
#pragma unroll
                        for (int r = 0; r < 4; ++r) {         // the plane's scale
                            const float sc = half_bits(parameter(pb, r, 0, j));
#pragma unroll
                            for (int nb = 0; nb < NB; ++nb) {
                                const int* v = &d[r >> 1][nb][2 * (r & 1)];
                                own[r >> 1][nb][r & 1] = fmaf(sc, (float)(v[0] + 256 * v[1]) * fac[nb], own[r >> 1][nb][r & 1]);
                            }
                        }
                    };
                    load_digits(0, 1.f);
#pragma unroll
                    for (int j = 0; j < Q; ++j) plane(j);
                    if (__builtin_expect(reinterpret_cast<const uint32_t*>(meta)[2 * MP] != 0u, 0)) {        // what the digits leave, in units 2^15 times smaller
                        load_digits(1, 0x1p-15f);
#pragma unroll 1
                        for (int j = 0; j < Q; ++j) plane(j);
                    }
                }
#pragma unroll
                for (int t = 0; t < 2; ++t)
#pragma unroll
                    for (int nb = 0; nb < NB; ++nb)
#pragma unroll
                        for (int i = 0; i < 2; ++i) acc[t][nb][i] += own[t][nb][i];
            }
            if constexpr (!BYTES) {
            if (step < steps_of(chunk0 + cu)) {
                const uint32_t wb = smem_addr(sW) + (uint32_t)(w.i * C::UNIT_BYTES);
                const uint32_t xb = smem_addr(sX) + (uint32_t)(x.i * XF_BYTES + step * (NB * 2048) + lane * 16);
                const float* meta = sM + x.i * XM_FLOATS + step * XM_STEP + 2 * c;
                uint4 xh[NB][4];                              // B fragments, held over the planes
#pragma unroll
                for (int nb = 0; nb < NB; ++nb)
#pragma unroll
                    for (int i = 0; i < 4; ++i) xh[nb][i] = lds128(xb + (uint32_t)((nb * 4 + i) * 512));
                float2 fac[NB];
#pragma unroll
                for (int nb = 0; nb < NB; ++nb) fac[nb] = *reinterpret_cast<const float2*>(meta + 8 * nb);
                // The step's sum is formed by itself where the registers allow it: in one chain over all chunks and planes the fp32
                // roundings add up (4096 x 14336, q = 4, G = 64, M = 8: 2.0e-7 of the result, 1.1e-7 so; the look-up kernel 1.2e-7).
                float own[kStepSum ? 2 : 1][kStepSum ? NB : 1][4];
                auto& sum = [&]() -> auto& {
                    if constexpr (kStepSum) return own;
                    else return acc;
                }();
                // offsets times the groups' activation sums
#pragma unroll
                for (int p = 0; p < NSG; ++p) {
                    float z[4];
#pragma unroll
                    for (int r = 0; r < 4; ++r) z[r] = half_bits(parameter(wb, r, p, Q) & offset_mask);
#pragma unroll
                    for (int nb = 0; nb < NB; ++nb) {
                        const float2 s = *reinterpret_cast<const float2*>(meta + (1 + p) * MP + 8 * nb);
#pragma unroll
                        for (int t = 0; t < 2; ++t)
#pragma unroll
                            for (int i = 0; i < 4; ++i) {
                                const float zi = z[2 * t + (i >> 1)], si = (i & 1) ? s.y : s.x;
                                sum[t][nb][i] = kStepSum && p == 0 ? zi * si : fmaf(zi, si, sum[t][nb][i]);
                            }
                    }
                }
                if (use_planes) {
#pragma unroll
                for (int j = 0; j < Q; ++j) {
                    uint32_t sub[2][4];                       // sub-words of the four rows
#pragma unroll
                    for (int r = 0; r < 4; ++r) {
                        const uint32_t tb = wb + (uint32_t)((r >> 1) * C::TILE_BYTES + j * 512);
                        if constexpr (G == 128) {
                            const uint32_t w0 = lds32(tb + off0[r & 1]), w1 = lds32(tb + off1[r & 1]);
                            sub[0][r] = __byte_perm(w0, w1, sel[0]);
                            sub[1][r] = __byte_perm(w0, w1, sel[1]);
                        } else {
#pragma unroll
                            for (int p = 0; p < 2; ++p) {
                                const uint32_t go = (uint32_t)(((p - (r & 1)) & 1) * 8);
                                sub[p][r] = __byte_perm(lds32(tb + off0[r & 1] + go), lds32(tb + off1[r & 1] + go), sel[0]);
                            }
                        }
                    }
                    float d[2][NB][4];
#pragma unroll
                    for (int q = 0; q < 2; ++q) {
                        if (q == 0 || NSG == 2) {
#pragma unroll
                            for (int t = 0; t < 2; ++t)
#pragma unroll
                                for (int nb = 0; nb < NB; ++nb)
#pragma unroll
                                    for (int i = 0; i < 4; ++i) d[t][nb][i] = 0.f;
                        }
#pragma unroll
                        for (int i2 = 0; i2 < 2; ++i2) {      // bits 4 i2 .. 4 i2 + 3 of the sub-word's bytes: two MMAs
                            uint32_t f[4][4];
#pragma unroll
                            for (int r = 0; r < 4; ++r) {
                                const uint32_t v = sub[q][r] * (i2 ? by64 : by4);
#pragma unroll
                                for (int i = 0; i < 4; ++i) f[r][i] = v & (0x04000400u << i);
                            }
#pragma unroll
                            for (int nb = 0; nb < NB; ++nb) {
                                const uint4 xv = xh[nb][2 * q + i2];
#pragma unroll
                                for (int t = 0; t < 2; ++t) {
                                    mma_16816(d[t][nb], f[2 * t][0], f[2 * t + 1][0], f[2 * t][1], f[2 * t + 1][1], xv.x, xv.y);
                                    mma_16816(d[t][nb], f[2 * t][2], f[2 * t + 1][2], f[2 * t][3], f[2 * t + 1][3], xv.z, xv.w);
                                }
                            }
                        }
                        if (q == 1 || NSG == 2) {             // the group is complete: its scale
                            const int p = NSG == 2 ? q : 0;
                            float sc[4];
#pragma unroll
                            for (int r = 0; r < 4; ++r) sc[r] = half_bits(parameter(wb, r, p, j));
#pragma unroll
                            for (int t = 0; t < 2; ++t)
#pragma unroll
                                for (int nb = 0; nb < NB; ++nb) {
                                    sum[t][nb][0] = fmaf(sc[2 * t], d[t][nb][0] * fac[nb].x, sum[t][nb][0]);
                                    sum[t][nb][1] = fmaf(sc[2 * t], d[t][nb][1] * fac[nb].y, sum[t][nb][1]);
                                    sum[t][nb][2] = fmaf(sc[2 * t + 1], d[t][nb][2] * fac[nb].x, sum[t][nb][2]);
                                    sum[t][nb][3] = fmaf(sc[2 * t + 1], d[t][nb][3] * fac[nb].y, sum[t][nb][3]);
                                }
                        }
                    }
                }
                }
                if constexpr (kStepSum) {
#pragma unroll
                    for (int t = 0; t < 2; ++t)
#pragma unroll
                        for (int nb = 0; nb < NB; ++nb)
#pragma unroll
                            for (int i = 0; i < 4; ++i) acc[t][nb][i] += sum[t][nb][i];
                }
            }
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(bar(kBarXEmpty + x.i));
            w.next();
            x.next();
            if (FOLD && (cu & 1)) {
#pragma unroll
                for (int nb = 0; nb < NB; ++nb)
#pragma unroll
                    for (int t = 0; t < 2; ++t)
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            own_sum[sum_at(nb, t, i)] = cu == 1 ? acc[t][nb][i] : own_sum[sum_at(nb, t, i)] + acc[t][nb][i];
                            acc[t][nb][i] = 0.f;
                        }
            }
        }

        // The four steps' sums meet in shared memory and are added and written out row by row.  (Where a warp gave up all leave
        // together: the barrier itself tells them, as a flag could be raised for the next run before every warp has read it for this one.)
        compute_sync();                                       // the buffer has been read; the ticket of the run before is there
        finish_tile(pending);
        pending = -1;
        if constexpr (BYTES) {                                // the upper digits' part
#pragma unroll
            for (int nb = 0; nb < NB; ++nb)
#pragma unroll
                for (int t = 0; t < 2; ++t)
#pragma unroll
                    for (int i = 0; i < 2; ++i) acc[t][nb][i] += __shfl_xor_sync(0xffffffffu, acc[t][nb][i], 1);
        }
        if (!BYTES || !(c & 1))
#pragma unroll
        for (int nb = 0; nb < NB; ++nb)
#pragma unroll
            for (int t = 0; t < 2; ++t)
#pragma unroll
                for (int i = 0; i < NE; ++i)
                    own_sum[sum_at(nb, t, i)] = FOLD && n_units > 1 ? own_sum[sum_at(nb, t, i)] + acc[t][nb][i] : acc[t][nb][i];
        if (compute_any(!live)) {                             // the tickets of this run of units and the rest are taken all the same
            gone = true;
            for (int v = u - n_units; v < u1 && tid == 0 && !SPLIT;) {
                const int t_ = a.by_chunks.of(v), end = min((t_ + 1) * C_, u1);
                if (end - v < C_) {
                    const unsigned t = atomicAdd(ticket_of(t_), 1u + kTicketNoPart);
                    if ((t & (kTicketNoPart - 1)) == (unsigned)(parts_of(t_) - 1)) *ticket_of(t_) = 0;
                }
                v = end;
            }
            break;
        }
        if constexpr (SPLIT) break;                           // (its only run: the cluster adds up)
        const int row = tid & (kUnitRows - 1), n = row_tile(tile) * kUnitRows + row, mb = batch0(tile), m_end = min(MP, M - mb);
        const bool whole = n_units == C_;
        float* part = a.g.partials + ((size_t)(b - a.by_cta.of(tile * C_)) * M + mb) * n_pad + n;
        for (int m = tid >> 7; m < m_end; m += kComputeThreads / kUnitRows) {
            const float y = sum_of(m, row, n, chunk0, chunk0 + n_units);
            if (whole) {
                if (n < N) put(mb + m, n, y);
            } else if ((size_t)n < n_pad) {
                part[(size_t)m * n_pad] = y;
            }
        }
        if (!whole) {                                         // a ticket; what it says is looked at after the next run of units
            compute_sync();
            if (tid == 0) {
                const int parts = parts_of(tile);
                unsigned t;                                   // (one operation that releases and acquires: between two fences it takes twice as long)
                asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], 1;" : "=r"(t) : "l"(ticket_of(tile)) : "memory");
                if ((t & (kTicketNoPart - 1)) == (unsigned)(parts - 1)) *ticket_of(tile) = 0;      // zero again for the next call
                *ticket_box = t == (unsigned)(parts - 1) ? 1u : 0u;
            }
            pending = tile;
        }
    }
    compute_sync();
    finish_tile(pending);
    if constexpr (SPLIT) {
        // The first CTA of the cluster adds the others' sums to its own, in ascending k order (and in pairs, as above), and writes them out.
        const int tile = b / a.split, row = tid & (kUnitRows - 1), n = row_tile(tile) * kUnitRows + row, mb = batch0(tile), m_end = min(MP, M - mb);
        __syncwarp();
        cluster_wait();                                       // the first CTA is there
        float y[MP / 4 + 1];
        if (gone) {
            if (tid == 0) st_cluster_u32((uint32_t)__cvta_generic_to_shared((const void*)lost_box), 0u, 1u);
        } else {
#pragma unroll
            for (int i = 0; i < (MP + 3) / 4; ++i) {
                const int m = (tid >> 7) + 4 * i;
                if (m >= m_end) continue;
                y[i] = sum_of(m, row, n, u0 - tile * C_, u1 - tile * C_);
                if (rank > 0) st_cluster_u32(smem_addr(sParts + ((rank - 1) * MP + m) * kUnitRows + row), 0u, __float_as_uint(y[i]));
            }
        }
        __syncwarp();
        cluster_arrive();
        cluster_wait();                                       // the parts are there
        if (rank == 0 && !gone && *lost_box == 0u && n < N) {
#pragma unroll
            for (int i = 0; i < (MP + 3) / 4; ++i) {
                const int m = (tid >> 7) + 4 * i;
                if (m >= m_end) continue;
                auto part = [&](int r) { return r == 0 ? y[i] : r < a.split ? sParts[((r - 1) * MP + m) * kUnitRows + row] : 0.f; };
                float sum = 0.f;
                for (int r = 0; r < a.split; r += 4) sum += (part(r) + part(r + 1)) + (part(r + 2) + part(r + 3));
                put(mb + m, n, sum);
            }
        }
    }
    __syncthreads();                                          // nobody leaves while copies are in flight
}

template <int Q, int G, int NB, bool BYTES, bool FOLD = false>
int launch_frag_cfg(const GemmArgs& g, int num_sms, cudaStream_t stream) {
    using C = FragCfg<Q, G>;
    constexpr int kMaxSmem = 232448, MP = (BYTES ? 2 : 8) * NB;
    constexpr int kFixed = kXSlots * (NB * 8192 + 4 * ((1 + C::NSG) * MP + (BYTES ? 1 : 0)) * 4) + 4 * MP * kSumStride * 4 + kNumBars * 8 + 64;
    static bool configured[64] = {};
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev >= 0 && dev < 64 && !configured[dev]) {
        cudaError_t e = cudaFuncSetAttribute(hlq_frag_kernel<Q, G, NB, FOLD, BYTES, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem);
        if (e == cudaSuccess) e = cudaFuncSetAttribute(hlq_frag_kernel<Q, G, NB, FOLD, BYTES, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem);
        if (e != cudaSuccess) return (int)e;
        configured[dev] = true;
    }
    FragArgs a;
    a.g = g;
    a.n_steps = (g.K + 127) / 128;
    a.chunks = g.n_kc;
    a.blocks = (g.M + MP - 1) / MP;
    const long long units = (long long)((g.N + kUnitRows - 1) / kUnitRows) * a.blocks * g.n_kc;
    if (units >= (1LL << 30)) return (int)cudaErrorInvalidValue;
    a.units = (int)units;
    a.per_cta = (a.units + num_sms - 1) / num_sms;
    // Few output tiles: each to a cluster of CTAs, where its longest share is no longer than equal runs of all units would be.  A ticket's round trip
    // through the L2, behind its fence, costs 1800 cycles and the parts as much again; the cluster's barriers and its writes to the first CTA's shared
    // memory about 1000.  (us, tickets / clusters: 4096 x 4096, M = 4, q = 2, 3, 4 6.8, 7.7, 8.8 / 6.1, 7.4, 8.7, M = 8 7.3, 8.3, 9.6 / 6.3, 7.4, 8.7; 4096 x 14336,
    // M = 8, q = 3 18.9 / 17.7; 5003 x 2880, G = 64, q = 3, M = 16 13.1 / 11.3.  A longer share loses: a unit more takes 0.5 + 0.6 q us.)
    // Of clusters of 3, 5 or 7 an eighth less than are resident together: behind a launch whose CTAs are still leaving, the last odd clusters
    // find no place and make a second wave (of 45 and 26 resident clusters of 3 and 5, from 43 and, after an idle chip, 24 on; even sizes, up to all
    // resident ones, never.  us, before there were clusters / with up to 45 / now: 1834 x 4416, G = 64, q = 4, M = 35 19.0 / 29.3 / 18.7; 3261 x 6784, q = 4,
    // M = 4, with 26 of five 14.7 / 16.7 / 14.4.  Up to 40 and 23 they are 2 to 16 % ahead of tickets behind every kernel tried.)
    a.split = 1;
    int longest = a.per_cta;
    if (a.per_cta < a.chunks) {
        const int tiles = a.units / a.chunks;
        for (int n = 2; n <= 8 && n <= a.chunks; ++n) {
            const int share = (a.chunks + n - 1) / n;
            const int most = resident_clusters(n) - (n % 2 ? resident_clusters(n) / 8 : 0);
            if (tiles <= most && (share < longest || (share == longest && a.split == 1))) {
                a.split = n;
                longest = share;
            }
        }
    }
    // Runs of more than two units without a sum per step: the sums are put by in between, for the same reason as there (4096 x 14336, q = 4,
    // G = 64, M = 16, error of the fp32 result 1.5e-7 -> 1.0e-7, the look-up kernel 1.0e-7 to 1.5e-7 by the number of rows; time
    // 36.3 -> 36.8 us).
    if constexpr (NB > 1 && !FOLD && !BYTES) {
        if (longest > 2) return launch_frag_cfg<Q, G, NB, BYTES, true>(g, num_sms, stream);
    }
    a.by_chunks.set(a.chunks);
    a.by_blocks.set(a.blocks);
    a.by_cta.set(a.per_cta);
    const int grid = a.split > 1 ? a.units / a.chunks * a.split : (a.units + a.per_cta - 1) / a.per_cta;
    const int parts_bytes = (a.split - 1) * MP * kUnitRows * 4;
    a.tickets = g.tickets;
    static_assert((kMaxSmem - kFixed - 7 * MP * kUnitRows * 4) / C::UNIT_BYTES >= 2, "shared memory");
    a.ws = (kMaxSmem - kFixed - parts_bytes) / C::UNIT_BYTES;
    if (a.ws > 5) a.ws = 5;

    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3(kFragThreads);
    cfg.dynamicSmemBytes = a.ws * C::UNIT_BYTES + kFixed + parts_bytes;
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = (unsigned)a.split;
    attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = a.split > 1 ? 2 : 1;
    cudaError_t e = cudaLaunchKernelEx(&cfg, a.split > 1 ? hlq_frag_kernel<Q, G, NB, FOLD, BYTES, true> : hlq_frag_kernel<Q, G, NB, FOLD, BYTES, false>, a);
    count_launch(1);
    return (int)e;
}

template <int Q, int G>
int launch_frag_qg(const GemmArgs& g, int num_sms, cudaStream_t stream) {
    // Up to four rows: as bytes (us as halves / bytes, M = 4, q = 2, 3, 4: 28672 x 4096 25.1, 31.6, 38.2 / 24.0, 29.4, 35.1; 4096 x 14336
    // 15.0, 18.5, 22.8 / 14.1, 17.3, 20.9; 4096 x 4096 7.4, 8.3, 9.5 / 7.2, 8.1, 9.1), but for three and four at q = 1, where preparing the
    // digits takes as long as the one plane (18.7, 11.1, 6.1 / 19.5, 11.5, 6.2; two rows at 4096 x 14336 9.0, on the look-up kernel 11.1).  At G = 64 the sums of a
    // step's two groups cost what the masks save (28672 x 4096, M = 4 27.6, 35.3, 43.0 / 28.7, 35.4, 41.5; 4096 x 4096 8.0, 9.4, 10.9 / 8.5, 9.9, 11.0).
    if constexpr (G == 128) {
        if (g.M <= 2) return launch_frag_cfg<Q, G, 1, true>(g, num_sms, stream);
        if constexpr (Q > 1) {
            if (g.M <= 4) return launch_frag_cfg<Q, G, 2, true>(g, num_sms, stream);
        }
    }
    if constexpr (G == 64) {
        // The height of a batch block, by the longest run of units: a unit takes u us, the first one of a taller block u0 more.  (Fitted
        // to 1100 calls, 256 to 28672 rows.  Blocks of 32 rows, whose sums do not fit the registers, are nowhere ahead: 4096 x 4096,
        // q = 4, M = 32 23.3 us in blocks of 16, 28.3 of 32; 28672 x 8192 218 and 232.)  A cluster's longest share is as long as the equal runs would be in all but a
        // few calls, so counting it instead changes no choice.  Since there are clusters, the choice is 2.9 % behind the better height over 400 calls of
        // 9 to 40 rows; 60 of them lose 5 % and more, most of these with one to three units a CTA (us, taken / other height: 499 x 7744, q = 3, M = 18
        // 12.3 / 7.6, in clusters of eight; 4264 x 576, q = 1, M = 39 7.5 / 5.2).
        const long long tiles = (long long)((g.N + kUnitRows - 1) / kUnitRows) * g.n_kc;
        auto us = [&](int rows, double u0, double u) {
            const long long units = tiles * ((g.M + rows - 1) / rows);
            return u0 + u * (double)((units + num_sms - 1) / num_sms);
        };
        if (g.M > 8 && us(16, 1.0, 1.0 + 0.86 * Q) < us(8, 0.0, 0.5 + 0.6 * Q)) return launch_frag_cfg<Q, G, 2, false>(g, num_sms, stream);
        return launch_frag_cfg<Q, G, 1, false>(g, num_sms, stream);
    }
    return g.M <= 8 ? launch_frag_cfg<Q, G, 1, false>(g, num_sms, stream) : (int)cudaErrorInvalidValue;
}

template <int Q>
int launch_frag_q(const GemmArgs& g, int G, int num_sms, cudaStream_t stream) {
    switch (G) {
        case 64: return launch_frag_qg<Q, 64>(g, num_sms, stream);
        case 128: return launch_frag_qg<Q, 128>(g, num_sms, stream);
        default: return (int)cudaErrorNotSupported;
    }
}

}  // namespace

// Up to ELUTQ_FRAGMENT_MAX_M rows at G = 128, any number at G = 64.
int launch_hlq_frag(const GemmArgs& g, int q, int G, int num_sms, cudaStream_t stream) {
    switch (q) {
        case 1: return launch_frag_q<1>(g, G, num_sms, stream);
        case 2: return launch_frag_q<2>(g, G, num_sms, stream);
        case 3: return launch_frag_q<3>(g, G, num_sms, stream);
        case 4: return launch_frag_q<4>(g, G, num_sms, stream);
        default: return (int)cudaErrorInvalidValue;
    }
}

}  // namespace elutq
