// Algorithm 1 on the GPU: alternating bit-pattern selection and least squares.
//
// The step before the hot path: it turns unquantised fp16 weights into the (B, s, z) that elutq_pack
// consumes.  Groups are independent.  Two forms with the same results bit for bit:
//
//   sorted   a lane per group.  The nearest candidate of a weight only depends on between which candidates it lies, so once
//            a group's weights are sorted a round needs the 2^q - 1 places where the choice changes, not a look at every
//            weight: a binary search on an estimate of each place, settled by the exact comparison of the two candidates at the
//            neighbouring weights; bit counts and right-hand sides follow from the places and prefix sums.  A lane sorts its group in its
//            registers, two weights in each (no shuffles: 1600 instructions for a warp's 32 groups of 128; a warp that sorts them two at a time
//            takes over 5000), runs its rounds, then the warp writes the bits.  A round's instructions are shared by 32 groups.  4096 x 4096, G = 128,
//            ten rounds, us: q = 2 688 direct (561 with the stop at unchanged bits), 112 sorted by the warp, 91 by lanes, 79 with a round's searches
//            side by side, 70 with the output's loads in flight; q = 4 2293 (1616), 611, 541, 517, 349 with its candidates in registers, 340.
//   direct   a warp per group (G / 32 weights per lane) that evaluates every candidate for every weight: for few groups, for the error
//            trace, and for groups with two candidates so close that rounding decides between them.
//
// The direct form:
//
//   initialisation   Delta = (max - min) / (2^q - 1), s = [Delta, 2 Delta, ...], z = min   (warp min / max)
//   selection        every lane evaluates the 2^q candidate values for its weights, first minimum wins
//   normal equations the matrix [B 1]^T [B 1] holds bit counts: ballots + popcounts, exact integers; the
//                    right-hand side sums weights in units of 2^-24 (every fp16 value is such an integer)
//                    in 64-bit integers, so the result does not depend on the reduction order
//   singular?        decided exactly by fraction-free elimination on the integer matrix; a singular system
//                    (a plane constant over the group, two equal planes) keeps the previous parameters
//   solve            elimination without pivoting and back substitution in fp64, one rounding per operation
//                    (explicit round-to-nearest intrinsics, no fused multiply-add), done redundantly by
//                    every lane
//
// All arithmetic that decides a bit is fp64 in a fixed order, so the selected planes and the fp16
// parameters are reproducible bit for bit.
#include "common.cuh"

namespace elutq {

namespace {

constexpr int kFitWarps = 8;      // warps (groups) per CTA
// From how many groups on the sorted form is taken, by the rounds asked for: 1, 2 to 4, 5 and more; in 1024 groups.  Its sort has to pay off over the rounds
// that a group runs.  With weights as trained layers have them it is ahead from a third to a half of these numbers on, but groups whose bits settle at once
// take the direct form two rounds, and those with candidates within rounding of each other are taken direct after all, the 32 of a warp in turn.  (us, direct /
// sorted, 4096, 8192 and 12288 groups of 128, ten rounds: q = 2, ordinary 28 / 20, 44 / 21, 62 / 21, on a grid of four values 6.7 / 9.2, 10 / 10, 14 / 10, of one value
// 6 / 44, 9 / 44, 13 / 44, of three 9.5 / 73, 14 / 73, 19 / 75; q = 4, ordinary 73 / 66, 125 / 74, 177 / 75, of sixteen values 29 / 43, 47 / 48, 66 / 49, of one 12 / 78, 20 / 79, 30 / 79.)
constexpr int kSortedMinK[3][4][3] = {{{12, 12, 16}, {12, 8, 8}, {12, 8, 12}, {12, 12, 24}},               // G = 32: q = 1 to 4
                                      {{32, 24, 16}, {24, 12, 12}, {12, 8, 8}, {12, 12, 16}},              // G = 64
                                      {{128, 64, 24}, {32, 24, 12}, {24, 12, 8}, {24, 12, 12}}};           // G = 128
inline long long sorted_min_groups(int q, int G, int t_max) {
    return 1024LL * kSortedMinK[G == 128 ? 2 : G == 64 ? 1 : 0][q - 1][t_max == 1 ? 0 : t_max < 5 ? 1 : 2];
}

__device__ __forceinline__ long long warp_sum_ll(long long v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
__device__ __forceinline__ double warp_sum_d(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = __dadd_rn(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

// The direct form for one group, by a whole warp.
template <int Q, int EPL>
__device__ __forceinline__ void fit_group(const __half* __restrict__ W, long long grp, long long n_groups, int t_max,
                                          uint8_t* __restrict__ planes, __half* __restrict__ scales, __half* __restrict__ offsets,
                                          double* __restrict__ trace) {
    constexpr int G = 32 * EPL, NC = 1 << Q, NV = Q + 1;
    const int lane = threadIdx.x & 31;
    const size_t base = (size_t)grp * G, plane_stride = (size_t)n_groups * G;      // (groups are contiguous: K is a multiple of G)

    double w[EPL];
    long long wfix[EPL];
    double wmax, wmin;
#pragma unroll
    for (int e = 0; e < EPL; ++e) {
        w[e] = (double)__half2float(W[base + lane + 32 * e]);
        wfix[e] = (long long)(w[e] * 16777216.0);          // exact: fp16 values are multiples of 2^-24
    }
    wmax = w[0];
    wmin = w[0];
#pragma unroll
    for (int e = 1; e < EPL; ++e) {
        wmax = fmax(wmax, w[e]);
        wmin = fmin(wmin, w[e]);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        wmax = fmax(wmax, __shfl_xor_sync(0xffffffffu, wmax, o));
        wmin = fmin(wmin, __shfl_xor_sync(0xffffffffu, wmin, o));
    }

    double s[Q], z = wmin;
    const double delta = __ddiv_rn(__dsub_rn(wmax, wmin), (double)(NC - 1));
#pragma unroll
    for (int j = 0; j < Q; ++j) s[j] = delta * (double)(1 << j);      // exact scaling

    int code[EPL], before[EPL];
#pragma unroll
    for (int e = 0; e < EPL; ++e) before[e] = -1;
    auto select = [&]() {
        double V[NC];
#pragma unroll
        for (int k = 0; k < NC; ++k) {
            double v = 0.0;
#pragma unroll
            for (int j = 0; j < Q; ++j)
                if ((k >> j) & 1) v = __dadd_rn(v, s[j]);
            V[k] = v;
        }
#pragma unroll
        for (int e = 0; e < EPL; ++e) {
            const double shifted = __dsub_rn(w[e], z);
            int best = 0;
            double bd = fabs(__dsub_rn(shifted, V[0]));
#pragma unroll
            for (int k = 1; k < NC; ++k) {
                const double d = fabs(__dsub_rn(shifted, V[k]));
                if (d < bd) { bd = d; best = k; }
            }
            code[e] = best;
        }
    };
    auto group_sse = [&]() {
        double acc = 0.0;
#pragma unroll
        for (int e = 0; e < EPL; ++e) {
            double rec = z;
#pragma unroll
            for (int j = 0; j < Q; ++j)
                if ((code[e] >> j) & 1) rec = __dadd_rn(rec, s[j]);
            const double d = __dsub_rn(w[e], rec);
            acc = __dadd_rn(acc, __dmul_rn(d, d));
        }
        return warp_sum_d(acc);
    };

    if (trace != nullptr) {
        select();
        const double e0 = group_sse();
        if (lane == 0) trace[grp] = e0;
    }

    for (int t = 1; t <= t_max; ++t) {
        select();
        // the same bits as in the round before: the parameters are theirs already, and so on in every later round
        bool same = true;
#pragma unroll
        for (int e = 0; e < EPL; ++e) {
            same &= code[e] == before[e];
            before[e] = code[e];
        }
        if (__all_sync(0xffffffffu, same)) {
            if (trace == nullptr) break;
            const double et = group_sse();
            if (lane == 0)
                for (int r = t; r <= t_max; ++r) trace[(size_t)r * n_groups + grp] = et;
            break;
        }

        // ---- normal equations: bit counts (exact) and fixed-point weight sums (exact) -----------------
        long long A[NV][NV];
        {
            unsigned mask[Q][EPL];
#pragma unroll
            for (int j = 0; j < Q; ++j)
#pragma unroll
                for (int e = 0; e < EPL; ++e) mask[j][e] = __ballot_sync(0xffffffffu, (code[e] >> j) & 1);
#pragma unroll
            for (int i = 0; i < Q; ++i) {
#pragma unroll
                for (int j = i; j < Q; ++j) {
                    int c = 0;
#pragma unroll
                    for (int e = 0; e < EPL; ++e) c += __popc(mask[i][e] & mask[j][e]);
                    A[i][j] = c;
                    A[j][i] = c;
                }
                int c = 0;
#pragma unroll
                for (int e = 0; e < EPL; ++e) c += __popc(mask[i][e]);
                A[i][Q] = c;
                A[Q][i] = c;
            }
            A[Q][Q] = G;
        }
        double r[NV];
        {
            long long all = 0;
#pragma unroll
            for (int e = 0; e < EPL; ++e) all += wfix[e];
            r[Q] = __ll2double_rn(warp_sum_ll(all)) / 16777216.0;
#pragma unroll
            for (int j = 0; j < Q; ++j) {
                long long part = 0;
#pragma unroll
                for (int e = 0; e < EPL; ++e) part += ((code[e] >> j) & 1) ? wfix[e] : 0;
                r[j] = __ll2double_rn(warp_sum_ll(part)) / 16777216.0;
            }
        }

        // ---- exact singularity test: fraction-free elimination, a zero pivot means a singular system -----
        bool singular = false;
        {
            long long m[NV][NV];
#pragma unroll
            for (int i = 0; i < NV; ++i)
#pragma unroll
                for (int j = 0; j < NV; ++j) m[i][j] = A[i][j];
            // The divisions are exact and the quotients (minors of a Gram matrix of 0/1 vectors of length <= 128)
            // stay below 128^5 < 2^36, so rounding numerator * (1 / prev) in fp64 (relative error < 2^-50)
            // returns the exact integer; the numerators stay below 2^57.
            double inv_prev = 1.0;
#pragma unroll
            for (int c = 0; c < NV; ++c) {
                singular = singular || (m[c][c] == 0);
                const long long piv = singular ? 1 : m[c][c];
#pragma unroll
                for (int i = c + 1; i < NV; ++i)
#pragma unroll
                    for (int j = c + 1; j < NV; ++j)
                        m[i][j] = __double2ll_rn(__ll2double_rn(m[i][j] * piv - m[i][c] * m[c][j]) * inv_prev);
                inv_prev = 1.0 / (double)piv;
            }
        }

        // ---- solve (fp64, elimination without pivoting, one rounding per operation) ------------------------
        if (!singular) {
            double a[NV][NV], b[NV], x[NV];
#pragma unroll
            for (int i = 0; i < NV; ++i) {
                b[i] = r[i];
#pragma unroll
                for (int j = 0; j < NV; ++j) a[i][j] = (double)A[i][j];
            }
#pragma unroll
            for (int c = 0; c < NV; ++c) {
#pragma unroll
                for (int i = c + 1; i < NV; ++i) {
                    const double f = __ddiv_rn(a[i][c], a[c][c]);
#pragma unroll
                    for (int j = c + 1; j < NV; ++j) a[i][j] = __dsub_rn(a[i][j], __dmul_rn(f, a[c][j]));
                    b[i] = __dsub_rn(b[i], __dmul_rn(f, b[c]));
                }
            }
#pragma unroll
            for (int i = NV - 1; i >= 0; --i) {
                double acc = b[i];
#pragma unroll
                for (int j = i + 1; j < NV; ++j) acc = __dsub_rn(acc, __dmul_rn(a[i][j], x[j]));
                x[i] = __ddiv_rn(acc, a[i][i]);
            }
#pragma unroll
            for (int j = 0; j < Q; ++j) s[j] = x[j];
            z = x[Q];
        }
        if (trace != nullptr) {
            const double et = group_sse();
            if (lane == 0) trace[(size_t)t * n_groups + grp] = et;
        }
    }

    // ---- results: one byte per bit (the input format of elutq_pack), fp16 parameters ----------------------
#pragma unroll
    for (int j = 0; j < Q; ++j)
#pragma unroll
        for (int e = 0; e < EPL; ++e) planes[j * plane_stride + base + lane + 32 * e] = (uint8_t)((code[e] >> j) & 1);
    if (lane < Q) {
        double v = s[0];
#pragma unroll
        for (int j = 1; j < Q; ++j) v = (lane == j) ? s[j] : v;
        scales[(size_t)grp * Q + lane] = __double2half(v);
    }
    if (lane == Q) offsets[grp] = __double2half(z);
}

template <int Q, int EPL>
__global__ void __launch_bounds__(kFitWarps * 32) hlq_fit_kernel(const __half* __restrict__ W, long long n_groups, int t_max,
                                                                 uint8_t* __restrict__ planes, __half* __restrict__ scales,
                                                                 __half* __restrict__ offsets, double* __restrict__ trace) {
    const long long grp = (long long)blockIdx.x * kFitWarps + (threadIdx.x >> 5);
    if (grp < n_groups) fit_group<Q, EPL>(W, grp, n_groups, t_max, planes, scales, offsets, trace);
}

constexpr int kSortWarps = 4;     // warps (of 32 groups) per CTA of the sorted form
// Bytes of a group's record: weight i of a warp's lanes lies at 64 i, so that each lane has half a bank of its own whatever it looks at.  The record
// bounds the warps on an SM, and with them the latencies hidden: prefix sums of every 8 weights instead of 4 took G = 128 from 146 to 113 us (q = 2,
// 4096 x 4096, sorted by the warp); at G = 32 the longer remainders cost more (1027 / 1083 us, q = 4).
__host__ __device__ constexpr int sorted_step(int G) { return G == 32 ? 4 : 8; }
__host__ __device__ constexpr int sorted_record(int G) { return 2 * G + 8 * (G / sorted_step(G) + 1); }

// Determinant of [B 1]^T [B 1] (bit counts of at most 128): minors of order 4 stay below 2^30 in every partial sum.
template <int NV>
__device__ __forceinline__ bool gram_singular(const int (&m)[NV][NV]) {
    if constexpr (NV == 2) {
        return m[0][0] * m[1][1] - m[0][1] * m[1][0] == 0;
    } else {
        // minors of the first two rows by column pair, then row by row
        int d2[NV][NV];
#pragma unroll
        for (int a = 0; a < NV; ++a)
#pragma unroll
            for (int b = a + 1; b < NV; ++b) d2[a][b] = m[0][a] * m[1][b] - m[0][b] * m[1][a];
        auto d3 = [&](int a, int b, int c) { return m[2][a] * d2[b][c] - m[2][b] * d2[a][c] + m[2][c] * d2[a][b]; };
        if constexpr (NV == 3) {
            return d3(0, 1, 2) == 0;
        } else if constexpr (NV == 4) {
            return m[3][0] * d3(1, 2, 3) - m[3][1] * d3(0, 2, 3) + m[3][2] * d3(0, 1, 3) - m[3][3] * d3(0, 1, 2) == 0;
        } else {
            auto d4 = [&](int a, int b, int c, int d) {
                return m[3][a] * d3(b, c, d) - m[3][b] * d3(a, c, d) + m[3][c] * d3(a, b, d) - m[3][d] * d3(a, b, c);
            };
            return (long long)m[4][0] * d4(1, 2, 3, 4) - (long long)m[4][1] * d4(0, 2, 3, 4) + (long long)m[4][2] * d4(0, 1, 3, 4) -
                   (long long)m[4][3] * d4(0, 1, 2, 4) + (long long)m[4][4] * d4(0, 1, 2, 3) == 0;
        }
    }
}

// (A plain load, so that the compiler keeps it behind the stores of what it reads.)
template <int IMM>
__device__ __forceinline__ __half lds_half(uint32_t addr) { return *reinterpret_cast<const __half*>(__cvta_shared_to_generic(addr + IMM)); }

__host__ __device__ constexpr int log2_of(int n) { return n > 1 ? 1 + log2_of(n / 2) : 0; }

template <int Q, int G>
__global__ void __launch_bounds__(kSortWarps * 32) hlq_fit_sorted_kernel(const __half* __restrict__ W, long long n_groups, int t_max,
                                                                         uint8_t* __restrict__ planes, __half* __restrict__ scales,
                                                                         __half* __restrict__ offsets, const bool aligned, const bool wide) {
    constexpr int NC = 1 << Q, NV = Q + 1, NB = 32 * G / 128, H = G / 2;     // NB: blocks of 128 weights of a warp's 32 groups
    constexpr int PS = sorted_step(G), REC = sorted_record(G), RES = 48;    // a group's sorted weights, and prefix sums of every PS of them; its result
    static_assert(16 + 2 * (NC - 1) <= RES && RES <= REC, "");
    extern __shared__ __align__(16) uint8_t smem[];
    const int lane = threadIdx.x & 31;
    uint8_t* recs = smem + (threadIdx.x >> 5) * (32 * REC);
    const long long grp0 = ((long long)blockIdx.x * kSortWarps + (threadIdx.x >> 5)) * 32;
    if (grp0 >= n_groups) return;
    __half* sorted = reinterpret_cast<__half*>(recs) + lane;      // weight i of the lane's group at 32 i: every lane has its bank (half a bank)
    double* pre = reinterpret_cast<double*>(recs + 64 * G) + lane;
    const long long total = n_groups * G, w0 = grp0 * G;          // weights in all; the warp's first
    const size_t plane_stride = (size_t)total;

    auto load4 = [&](int block, __half (&h)[4]) {                 // weights 4 lane .. 4 lane + 3 of a block (zeros behind the end)
        const long long i = w0 + block * 128 + 4 * lane;
        if (aligned && i < total) {                               // (G is a multiple of 32: four weights are inside or outside)
            const uint2 r = *reinterpret_cast<const uint2*>(W + i);
            *reinterpret_cast<uint2*>(h) = r;
        } else {
#pragma unroll
            for (int e = 0; e < 4; ++e) h[e] = i + e < total ? W[i + e] : __ushort_as_half(0);
        }
    };

    // ---- sort: a lane its group, in registers.  Both halves of the registers are runs of their own, sorted by one network (Batcher's
    // odd-even merges) and then merged. ------------------------------------------------------------------------------------------
    const long long grp = grp0 + lane;
    const bool valid = grp < n_groups;
    {
        __half2 v[H];
        const __half* src = W + grp * G;
        if (wide) {
#pragma unroll
            for (int i = 0; i < H; i += 4) {
                const uint4 r = valid ? __ldg(reinterpret_cast<const uint4*>(src + 2 * i)) : make_uint4(0, 0, 0, 0);
                *reinterpret_cast<uint4*>(&v[i]) = r;
            }
        } else {
#pragma unroll
            for (int i = 0; i < H; ++i) v[i] = valid ? __halves2half2(src[2 * i], src[2 * i + 1]) : __float2half2_rn(0.f);
        }
        auto exchange = [&](int a, int b) {
            const __half2 mn = __hmin2(v[a], v[b]), mx = __hmax2(v[a], v[b]);
            v[a] = mn;
            v[b] = mx;
        };
        static_for<0, log2_of(H)>([&](auto p_c) {
            constexpr int p = 1 << decltype(p_c)::value;
            static_for<0, decltype(p_c)::value + 1>([&](auto k_c) {
                constexpr int k = p >> decltype(k_c)::value;
#pragma unroll
                for (int j = k % p; j <= H - 1 - k; j += 2 * k)
#pragma unroll
                    for (int i = 0; i < k; ++i)
                        if (i + j + k < H && (i + j) / (2 * p) == (i + j + k) / (2 * p)) exchange(i + j, i + j + k);
            });
        });
        // the lower halves against the upper ones in reverse: the smaller ones are the lower half of the result, and bitonic
#pragma unroll
        for (int i = 0; i < H / 2; ++i) {
            const int j = H - 1 - i;
            const __half2 o = __lowhigh2highlow(v[j]), mn = __hmin2(v[i], o), mx = __hmax2(v[i], o);
            v[i] = __lows2half2(mn, mx);
            v[j] = __highs2half2(mn, mx);
        }
#pragma unroll
        for (int k = H / 2; k >= 1; k >>= 1)
#pragma unroll
            for (int i = 0; i < H; ++i)
                if (!(i & k)) exchange(i, i + k);
        // sums of fp16 values are exact in fp64
        double run = 0.0;
#pragma unroll
        for (int i = 0; i < G; ++i) {
            const __half w = i < H ? __low2half(v[i % H]) : __high2half(v[i % H]);
            if (i % PS == 0) pre[i / PS * 32] = run;
            run += (double)__half2float(w);
            sorted[i * 32] = w;
        }
        pre[G / PS * 32] = run;
    }

    // ---- rounds: lane = group --------------------------------------------------------------------------------------------------
    auto weight = [&](int i) { return __half2float(sorted[i * 32]); };
    const uint32_t sorted_at = (uint32_t)__cvta_generic_to_shared(sorted);
    const double wmin = (double)weight(0), wmax = (double)weight(G - 1);
    double s[Q], z = wmin;
    const double delta = __ddiv_rn(__dsub_rn(wmax, wmin), (double)(NC - 1));
#pragma unroll
    for (int j = 0; j < Q; ++j) s[j] = delta * (double)(1 << j);      // exact scaling

    int cut[NC - 1];                                              // first weight above the r-th place
#pragma unroll
    for (int r = 0; r < NC - 1; ++r) cut[r] = -1;
    unsigned long long map = 0;                                   // nibble r: code of the r-th smallest candidate
    bool active = valid, direct = false;
    for (int t = 1; t <= t_max && __any_sync(0xffffffffu, active); ++t) {
        if (!active) continue;
        double V[NC];
        int code[NC];
#pragma unroll
        for (int k = 0; k < NC; ++k) {
            double v = 0.0;
#pragma unroll
            for (int j = 0; j < Q; ++j)
                if ((k >> j) & 1) v = __dadd_rn(v, s[j]);
            V[k] = v;
            code[k] = k;
        }
        // candidates in ascending order (odd-even merge exchanges)
        static_for<0, Q>([&](auto p_c) {                          // (unrolled for certain: the indices are constants)
            constexpr int p = 1 << decltype(p_c)::value;
            static_for<0, decltype(p_c)::value + 1>([&](auto k_c) {
                constexpr int k = p >> decltype(k_c)::value;
                static_for<0, NC - k>([&](auto x_c) {
                    constexpr int x = decltype(x_c)::value, y = x + k;
                    if constexpr ((x - k % p + 2 * k) % (2 * k) < k && x >= k % p && x / (2 * p) == y / (2 * p)) {
                        const bool swap = V[y] < V[x];
                        const double lo = swap ? V[y] : V[x], hi = swap ? V[x] : V[y];
                        const int cl = swap ? code[y] : code[x], ch = swap ? code[x] : code[y];
                        V[x] = lo;
                        V[y] = hi;
                        code[x] = cl;
                        code[y] = ch;
                    }
                });
            });
        });
        // Only the two candidates around a weight are in question as long as no two are within rounding of each other.
        const double gap = 9.094947017729282e-13 /* 2^-40 */ * (fmax(fabs(wmin), fabs(wmax)) + fabs(z) + fmax(fabs(V[0]), fabs(V[NC - 1])));
        bool apart = true;
#pragma unroll
        for (int r = 0; r < NC - 1; ++r) apart &= V[r + 1] - V[r] > gap;
        if (!apart) {                                             // (also for values that are not finite)
            direct = true;
            active = false;
            continue;
        }
        unsigned long long new_map = 0;
#pragma unroll
        for (int r = 0; r < NC; ++r) new_map |= (unsigned long long)code[r] << (4 * r);
        bool changed = new_map != map;
        map = new_map;
        // The places: a search on estimates of them, all side by side, and where a neighbouring weight is not clearly on its side, by the exact choice.
        // (An estimate is off by its rounding to fp32, the choice's own roundings are far below `gap`.)
        float guess[NC - 1];
        __half guess_up[NC - 1];                                  // (a weight is below the one where it is below the other)
        uint32_t at[NC - 1];                                      // where the place's weight lies: 64 bytes a weight
        int pos[NC - 1];
#pragma unroll
        for (int r = 0; r < NC - 1; ++r) {
            guess[r] = (float)(z + 0.5 * (V[r] + V[r + 1]));
            guess_up[r] = __float2half_ru(guess[r]);
            at[r] = sorted_at;
        }
        static_for<0, log2_of(G)>([&](auto i_c) {
            constexpr int st = G >> (decltype(i_c)::value + 1);
#pragma unroll
            for (int r = 0; r < NC - 1; ++r)
                if (__hlt(lds_half<64 * (st - 1)>(at[r]), guess_up[r])) at[r] += 64 * st;
        });
        const float gap_up = __double2float_ru(gap);
        bool clear = true;
#pragma unroll
        for (int r = 0; r < NC - 1; ++r) {
            if (__hlt(lds_half<0>(at[r]), guess_up[r])) at[r] += 64;
            const float near = fabsf(guess[r]) * 0x1p-22f + gap_up;
            const float below = __half2float(lds_half<0>(max(at[r] - 64, sorted_at))), above = __half2float(lds_half<0>(min(at[r], sorted_at + 64 * (G - 1))));
            clear &= at[r] == sorted_at || guess[r] - below > near;
            clear &= at[r] == sorted_at + 64 * G || above - guess[r] > near;
            pos[r] = (int)(at[r] - sorted_at) / 64;
        }
        if (!clear) {
#pragma unroll
            for (int r = 0; r < NC - 1; ++r) {
                auto above = [&](int i) {                         // the exact choice between candidates r and r + 1
                    const double shifted = __dsub_rn((double)weight(i), z);
                    const double da = fabs(__dsub_rn(shifted, V[r])), db = fabs(__dsub_rn(shifted, V[r + 1]));
                    return db < da || (db == da && code[r + 1] < code[r]);
                };
                while (pos[r] > 0 && above(pos[r] - 1)) --pos[r];
                while (pos[r] < G && !above(pos[r])) ++pos[r];
            }
        }
#pragma unroll
        for (int r = 0; r < NC - 1; ++r) {
            changed |= pos[r] != cut[r];
            cut[r] = pos[r];
        }
        // the same bits as in the round before: the parameters are theirs already, and so on in every later round
        if (!changed) {
            active = false;
            continue;
        }
        int A[NV][NV];
        double b[NV];
#pragma unroll
        for (int i = 0; i < NV; ++i) {
            b[i] = 0.0;
#pragma unroll
            for (int j = 0; j < NV; ++j) A[i][j] = 0;
        }
        A[Q][Q] = G;
        b[Q] = 0.0 + pre[G / PS * 32];                                // (never a negative zero)
        {
            int from = 0;
            double below = 0.0;
#pragma unroll
            for (int r = 0; r < NC; ++r) {
                const int to = r < NC - 1 ? cut[r < NC - 1 ? r : 0] : G;
                double upto = pre[to / PS * 32];
                if (r < NC - 1) {                                 // (exact in any order; what lies behind the place is read and left out)
                    double w[PS];
#pragma unroll
                    for (int e = 0; e < PS - 1; ++e) {
                        const double v = (double)weight(to / PS * PS + e);
                        w[e] = e < to % PS ? v : 0.0;
                    }
                    w[PS - 1] = upto;
#pragma unroll
                    for (int o = PS / 2; o > 0; o >>= 1)
#pragma unroll
                        for (int e = 0; e < o; ++e) w[e] += w[e + o];
                    upto = w[0];
                }
                const int cnt = to - from;
                const double part = upto - below;                 // exact
                from = to;
                below = upto;
#pragma unroll
                for (int i = 0; i < Q; ++i) {
                    if ((code[r] >> i) & 1) {
                        b[i] += part;
                        A[i][Q] += cnt;
                    }
#pragma unroll
                    for (int j = i; j < Q; ++j)
                        if (((code[r] >> i) & (code[r] >> j)) & 1) A[i][j] += cnt;
                }
            }
#pragma unroll
            for (int i = 0; i < NV; ++i)
#pragma unroll
                for (int j = 0; j < i; ++j) A[i][j] = A[j][i];
        }
        // fp64, elimination without pivoting, one rounding per operation (the direct form's order)
        if (!gram_singular(A)) {
            double a[NV][NV], x[NV];
#pragma unroll
            for (int i = 0; i < NV; ++i)
#pragma unroll
                for (int j = 0; j < NV; ++j) a[i][j] = (double)A[i][j];
#pragma unroll
            for (int c = 0; c < NV; ++c) {
#pragma unroll
                for (int i = c + 1; i < NV; ++i) {
                    const double f = __ddiv_rn(a[i][c], a[c][c]);
#pragma unroll
                    for (int j = c + 1; j < NV; ++j) a[i][j] = __dsub_rn(a[i][j], __dmul_rn(f, a[c][j]));
                    b[i] = __dsub_rn(b[i], __dmul_rn(f, b[c]));
                }
            }
#pragma unroll
            for (int i = NV - 1; i >= 0; --i) {
                double acc = b[i];
#pragma unroll
                for (int j = i + 1; j < NV; ++j) acc = __dsub_rn(acc, __dmul_rn(a[i][j], x[j]));
                x[i] = __ddiv_rn(acc, a[i][i]);
            }
#pragma unroll
            for (int j = 0; j < Q; ++j) s[j] = x[j];
            z = x[Q];
        }
    }

    // ---- results: parameters by lane; per group the weights at the places and the codes, then the bits by the warp -----------
    __half place[NC - 1];
#pragma unroll
    for (int r = 0; r < NC - 1; ++r) place[r] = cut[r] < G ? sorted[max(cut[r], 0) * 32] : __ushort_as_half(0x7c00);      // (infinity: none)
    __syncwarp();
    uint8_t* rec = recs + lane * RES;
    __half* places = reinterpret_cast<__half*>(rec + 16);
#pragma unroll
    for (int r = 0; r < NC; ++r) rec[r] = (uint8_t)(map >> (4 * r) & 15u);
#pragma unroll
    for (int r = 0; r < NC - 1; ++r) places[r] = place[r];
    if (valid && !direct) {
#pragma unroll
        for (int j = 0; j < Q; ++j) scales[(size_t)grp * Q + j] = __double2half(s[j]);
        offsets[grp] = __double2half(z);
    }
    const unsigned directs = __ballot_sync(0xffffffffu, direct);
    __syncwarp();
    auto put_bits = [&](int blk, const __half (&h)[4]) {
        const int g = (blk * 128 + 4 * lane) / G;
        const long long i = w0 + blk * 128 + 4 * lane;
        const uint8_t* gr = recs + g * RES;
        const __half* pl = reinterpret_cast<const __half*>(gr + 16);
        const uint4 cw = *reinterpret_cast<const uint4*>(gr);     // code of every rank, a byte each
        const uint32_t codes[4] = {cw.x, cw.y, cw.z, cw.w};
        __half2 rank[2] = {__float2half2_rn(1024.f), __float2half2_rn(1024.f)};      // (1024 + rank: the rank in the low bits)
        const __half2 w2[2] = {__halves2half2(h[0], h[1]), __halves2half2(h[2], h[3])};
#pragma unroll
        for (int r = 0; r < NC - 1; ++r) {
            const __half2 p2 = __half2half2(pl[r]);
            rank[0] = __hadd2(rank[0], __hge2(w2[0], p2));
            rank[1] = __hadd2(rank[1], __hge2(w2[1], p2));
        }
        // the ranks as the nibbles of a selector, the codes of the four weights as bytes
        const uint32_t r0 = *reinterpret_cast<const uint32_t*>(&rank[0]), r1 = *reinterpret_cast<const uint32_t*>(&rank[1]);
        const uint32_t lows = __byte_perm(r0, r1, 0x6420) & 0x0f0f0f0fu, sel = lows | lows >> 4;       // bytes: ranks; nibbles 0, 1, 4, 5 of sel
        const uint32_t pick = __byte_perm(sel, 0u, 0x4420);
        uint32_t four;
        if constexpr (Q <= 3) {
            four = __byte_perm(codes[0], codes[1], pick);
        } else {                                                  // ranks of 8 and more in the upper half
            const uint32_t lo = __byte_perm(codes[0], codes[1], pick & 0x7777u), hi = __byte_perm(codes[2], codes[3], pick & 0x7777u);
            const uint32_t upper = (lows >> 3 & 0x01010101u) * 0xffu;
            four = (lo & ~upper) | (hi & upper);
        }
        if (i < total && !((directs >> g) & 1u)) {
#pragma unroll
            for (int j = 0; j < Q; ++j) {
                const uint32_t bits = (four >> j) & 0x01010101u;
                uint8_t* dst = planes + j * plane_stride + i;
                if (aligned) {
                    *reinterpret_cast<uint32_t*>(dst) = bits;
                } else {
#pragma unroll
                    for (int e = 0; e < 4; ++e) dst[e] = (uint8_t)(bits >> (8 * e));
                }
            }
        }
    };
    if (aligned) {                                                // a few blocks' weights on their way at a time
        constexpr int kAhead = Q <= 2 ? 8 : Q == 3 ? 4 : G == 128 ? 2 : 1;      // (more of the longer code costs instruction fetches)
        static_assert(NB % kAhead == 0, "");
#pragma unroll 1
        for (int blk = 0; blk < NB; blk += kAhead) {
            uint2 raw[kAhead];
#pragma unroll
            for (int a = 0; a < kAhead; ++a) {
                const long long i = w0 + (blk + a) * 128 + 4 * lane;
                raw[a] = i < total ? __ldg(reinterpret_cast<const uint2*>(W + i)) : make_uint2(0, 0);
            }
#pragma unroll
            for (int a = 0; a < kAhead; ++a) put_bits(blk + a, reinterpret_cast<const __half (&)[4]>(raw[a]));
        }
    } else {
#pragma unroll 1
        for (int blk = 0; blk < NB; ++blk) {
            __half h[4];
            load4(blk, h);
            put_bits(blk, h);
        }
    }
    for (unsigned left = directs; left != 0; left &= left - 1)
        fit_group<Q, G / 32>(W, grp0 + __ffs(left) - 1, n_groups, t_max, planes, scales, offsets, nullptr);
}

template <int Q, int G>
int launch_fit_qg(const __half* W, int N, int K, int t_max, uint8_t* planes, __half* scales, __half* offsets, double* trace,
                  cudaStream_t stream) {
    const long long n_groups = (long long)N * (K / G);
    if (trace == nullptr && n_groups >= sorted_min_groups(Q, G, t_max)) {
        constexpr int kSmem = kSortWarps * 32 * sorted_record(G);
        static bool configured[64] = {};
        int dev = 0;
        cudaGetDevice(&dev);
        if (dev >= 0 && dev < 64 && !configured[dev]) {
            cudaError_t e = cudaFuncSetAttribute(hlq_fit_sorted_kernel<Q, G>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem);
            if (e != cudaSuccess) return (int)e;
            configured[dev] = true;
        }
        const bool aligned = ((reinterpret_cast<uintptr_t>(W) & 7) | (reinterpret_cast<uintptr_t>(planes) & 3)) == 0;
        const unsigned grid = (unsigned)((n_groups + 32 * kSortWarps - 1) / (32 * kSortWarps));
        hlq_fit_sorted_kernel<Q, G><<<grid, kSortWarps * 32, kSmem, stream>>>(W, n_groups, t_max, planes, scales, offsets, aligned, (reinterpret_cast<uintptr_t>(W) & 15) == 0);
    } else {
        const unsigned grid = (unsigned)((n_groups + kFitWarps - 1) / kFitWarps);
        hlq_fit_kernel<Q, G / 32><<<grid, kFitWarps * 32, 0, stream>>>(W, n_groups, t_max, planes, scales, offsets, trace);
    }
    count_launch(1);
    return (int)cudaGetLastError();
}

template <int Q>
int launch_fit_q(const __half* W, int G, int N, int K, int t_max, uint8_t* planes, __half* scales, __half* offsets,
                 double* trace, cudaStream_t stream) {
    switch (G) {
        case 32: return launch_fit_qg<Q, 32>(W, N, K, t_max, planes, scales, offsets, trace, stream);
        case 64: return launch_fit_qg<Q, 64>(W, N, K, t_max, planes, scales, offsets, trace, stream);
        case 128: return launch_fit_qg<Q, 128>(W, N, K, t_max, planes, scales, offsets, trace, stream);
        default: return (int)cudaErrorInvalidValue;
    }
}

}  // namespace

}  // namespace elutq

using namespace elutq;

extern "C" int elutq_hlq_fit(const void* W, int q, int G, int N, int K, int t_max, uint8_t* planes, void* scales,
                             void* offsets, double* err_trace, void* stream) {
    if (!W || !planes || !scales || !offsets) return ELUTQ_ERR_INVALID_ARG;
    if (N <= 0 || K <= 0 || t_max < 1 || t_max > 1000) return ELUTQ_ERR_INVALID_ARG;
    if (q < 1 || q > 4 || (G != 32 && G != 64 && G != 128) || K % G != 0) return ELUTQ_ERR_SHAPE;
    if ((reinterpret_cast<uintptr_t>(W) & 1) || (reinterpret_cast<uintptr_t>(scales) & 1) ||
        (reinterpret_cast<uintptr_t>(offsets) & 1) || (reinterpret_cast<uintptr_t>(err_trace) & 7))
        return ELUTQ_ERR_ALIGN;
    const __half* w = reinterpret_cast<const __half*>(W);
    __half* s = reinterpret_cast<__half*>(scales);
    __half* z = reinterpret_cast<__half*>(offsets);
    cudaStream_t st = (cudaStream_t)stream;
    int ce;
    switch (q) {
        case 1: ce = launch_fit_q<1>(w, G, N, K, t_max, planes, s, z, err_trace, st); break;
        case 2: ce = launch_fit_q<2>(w, G, N, K, t_max, planes, s, z, err_trace, st); break;
        case 3: ce = launch_fit_q<3>(w, G, N, K, t_max, planes, s, z, err_trace, st); break;
        default: ce = launch_fit_q<4>(w, G, N, K, t_max, planes, s, z, err_trace, st); break;
    }
    if (ce != 0) {
        note_cuda_error(ce);
        return ELUTQ_ERR_CUDA;
    }
    return ELUTQ_OK;
}
