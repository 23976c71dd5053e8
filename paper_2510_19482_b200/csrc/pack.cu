// Offline packing of HLQ bit-planes, scales and offsets into the device layout, and its inverse.
//
// Packing: a warp owns 32 plane vectors of 16 bytes of the output, a thread a 32-bit parameter word.
// Unpacking runs per logical element.  Neither is on the per-token path.
#include "common.cuh"

namespace elutq {

namespace {

__device__ __forceinline__ uint32_t header_word(const Geo& g, int i) {
    switch (i) {
        case 0: return (uint32_t)kMagic;
        case 1: return (uint32_t)kVersion;
        case 2: return (uint32_t)g.q;
        case 3: return (uint32_t)g.G;
        case 4: return (uint32_t)g.N;
        case 5: return (uint32_t)g.K;
        case 6: return (uint32_t)g.n_rb;
        case 7: return (uint32_t)g.n_kc;
        case 8: return (uint32_t)g.tile_bytes;
        default: return 0u;
    }
}

// Bit b of the result: byte b of x is not zero.
__device__ __forceinline__ uint32_t nonzero_bytes(uint32_t x) {
    // the bytes' top bits from any bit below them, then the four together: copies shifted by 7, 14, 21, 28 do not overlap
    const uint32_t m = ((((x & 0x7f7f7f7fu) + 0x7f7f7f7fu) | x) >> 7) & 0x01010101u;
    return (m * 0x10204080u) >> 28;
}

constexpr int kPackWarps = 8;

// One warp per 32 plane vectors of a tile: (tile, vec = u*q + j), 16 rows x 2 super-groups of 128 input bytes.  A load covers whole
// lines (four rows' 128 bytes), the bits go through shared memory to their places in the rows' rotated order, and the lanes store
// 16 bytes each.  (A thread per vector with sixteen loads of 8 bytes 128 bytes apart, and the order's divisions at run time: 4096 x 4096,
// q = 2 22 us.)
template <int Q, int G>
__device__ __forceinline__ void pack_plane_vectors(const uint8_t* __restrict__ planes, uint8_t* __restrict__ tiles, const Geo& g, int tile, int kc, int vec,
                                                   int lane, bool wide, uint8_t* place) {
    constexpr int W = G / 8, NSG = 128 / G;
    const int rb = tile - kc * g.n_rb, u = vec / Q, j = vec - u * Q;
    const int col = 2 * (lane & 7);                               // the lane's 16 input bytes: byte columns col, col + 1 of a super-group
    uint4 x[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const int seg = 4 * i + (lane >> 3), n = rb * kTileRows + (seg & 15), k0 = kc * kChunkK + ((seg >> 4) + 2 * u) * 128 + col * 8;
        const uint8_t* src = planes + ((size_t)j * g.N + n) * g.K + k0;
        x[i] = make_uint4(0u, 0u, 0u, 0u);
        if (n < g.N && k0 < g.K) {
            if (wide) {
                x[i] = __ldg(reinterpret_cast<const uint4*>(src));
            } else {
                const uint2 lo = __ldg(reinterpret_cast<const uint2*>(src)), hi = __ldg(reinterpret_cast<const uint2*>(src) + 1);
                x[i] = make_uint4(lo.x, lo.y, hi.x, hi.y);
            }
        }
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const int seg = 4 * i + (lane >> 3), l = seg & 15;
        const uint32_t bits[2] = {nonzero_bytes(x[i].x) | nonzero_bytes(x[i].y) << 4, nonzero_bytes(x[i].z) | nonzero_bytes(x[i].w) << 4};
#pragma unroll
        for (int e = 0; e < 2; ++e) {                             // the inverse of tau(l, i)
            const int c = col + e, at = ((c / W - l / W) & (NSG - 1)) * W + ((c - l) & (W - 1));
            place[seg * 16 + at] = (uint8_t)bits[e];
        }
    }
    __syncwarp();
    reinterpret_cast<uint4*>(tiles + (size_t)tile * g.tile_bytes)[vec * 32 + lane] = reinterpret_cast<const uint4*>(place)[lane];
}

// One thread per parameter word: (tile, word, lane) -> two fp16 values of the lane's record.
template <int Q, int G>
__device__ __forceinline__ void pack_param_word(const uint16_t* __restrict__ scales, const uint16_t* __restrict__ offsets,
                                                uint8_t* __restrict__ tiles, const Geo& g, int tile, int kc, int word, int lane) {
    constexpr int W = G / 8, NSG = 128 / G;
    const int rb = tile - kc * g.n_rb;
    const int h = lane >> 4, l = lane & 15;
    const int n = rb * kTileRows + l;
    const int Gn = g.K / G;
    const int a = l / W;
    uint32_t packed = 0;
#pragma unroll
    for (int half = 0; half < 2; ++half) {
        const int e = 2 * word + half;
        const int uv = e / (Q + 1), comp = e - uv * (Q + 1);
        const int u = uv / NSG, v = uv % NSG;
        const int gamma = NSG * (h + 2 * u) + (a + v) % NSG;      // group inside the chunk
        const int gi = kc * (kChunkK / G) + gamma;
        uint32_t bits = 0;
        if (n < g.N && gi < Gn) bits = comp < Q ? scales[((size_t)n * Gn + gi) * Q + comp] : offsets[(size_t)n * Gn + gi];
        packed |= bits << (16 * half);
    }
    reinterpret_cast<uint32_t*>(tiles + (size_t)tile * g.tile_bytes + g.plane_bytes)[word * 32 + lane] = packed;
}

// The whole blob in one launch: plane vectors, parameter words (blocks from plane_blocks on), the header.
template <int Q, int G>
__global__ void __launch_bounds__(32 * kPackWarps) pack_kernel(const uint8_t* __restrict__ planes, const uint16_t* __restrict__ scales,
                                                               const uint16_t* __restrict__ offsets, uint8_t* __restrict__ packed, const Geo g,
                                                               const int plane_blocks, const Div by_rows, const bool wide) {
    constexpr int kVectors = 2 * Q, kWords = 2 * (128 / G) * (Q + 1) / 2;        // warps' works of a tile
    __shared__ __align__(16) uint8_t place[kPackWarps][512];
    uint8_t* tiles = packed + ELUTQ_HEADER_BYTES;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const bool params = (int)blockIdx.x >= plane_blocks;
    const int i = ((int)blockIdx.x - (params ? plane_blocks : 0)) * kPackWarps + warp, per = params ? kWords : kVectors;
    const int tile = i / per, kc = by_rows.of(tile);
    if (tile < g.n_kc * g.n_rb) {
        if (params) pack_param_word<Q, G>(scales, offsets, tiles, g, tile, kc, i - tile * per, lane);
        else pack_plane_vectors<Q, G>(planes, tiles, g, tile, kc, i - tile * per, lane, wide, place[warp]);
    }
    if (params && i == 0 && lane < ELUTQ_HEADER_BYTES / 4) reinterpret_cast<uint32_t*>(packed)[lane] = header_word(g, lane);
}

// One thread per (plane j, row n, byte-column cg): expands a packed byte to 8 uint8 {0,1}.
__global__ void unpack_planes_kernel(const uint8_t* __restrict__ tiles, uint8_t* __restrict__ planes, Geo g) {
    if (!blob_header_matches(tiles, g.q, g.G, g.N, g.K, nullptr)) return;   // before any tile is read
    const int cols = g.K / 8;
    const long long total = (long long)g.q * g.N * cols;
    const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= total) return;
    const int cg = (int)(idx % cols);
    const int n = (int)((idx / cols) % g.N);
    const int j = (int)(idx / ((long long)cols * g.N));
    const int rb = n / kTileRows, l = n % kTileRows;
    const int kc = cg / 64, c = cg % 64;
    const int sigma = c / 16, tau = c % 16;
    const int h = sigma & 1, u = sigma >> 1;
    const int sg = tau / g.w, rr = tau % g.w;
    const int a = l / g.w, r = l % g.w;
    const int v = (sg - a + g.nsg) % g.nsg;
    const int ii = (rr - r + g.w) % g.w;
    const int i = v * g.w + ii;
    const size_t off = ((size_t)kc * g.n_rb + rb) * g.tile_bytes + ((size_t)(u * g.q + j) * 32 + 16 * h + l) * 16 + i;
    const uint32_t byte = tiles[off];
    uint64_t x = 0;
#pragma unroll
    for (int b = 0; b < 8; ++b) x |= (uint64_t)((byte >> b) & 1u) << (8 * b);
    *reinterpret_cast<uint64_t*>(planes + ((size_t)j * g.N + n) * g.K + (size_t)cg * 8) = x;
}

// One thread per (row n, group gi, component): copies one fp16 parameter back.
__global__ void unpack_params_kernel(const uint8_t* __restrict__ tiles, uint16_t* __restrict__ scales,
                                     uint16_t* __restrict__ offsets, Geo g) {
    if (!blob_header_matches(tiles, g.q, g.G, g.N, g.K, nullptr)) return;   // before any tile is read
    const int Gn = g.K / g.G;
    const long long total = (long long)g.N * Gn * (g.q + 1);
    const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= total) return;
    const int comp = (int)(idx % (g.q + 1));
    const int gi = (int)((idx / (g.q + 1)) % Gn);
    const int n = (int)(idx / ((long long)(g.q + 1) * Gn));
    const int rb = n / kTileRows, l = n % kTileRows;
    const int gpc = kChunkK / g.G;
    const int kc = gi / gpc, gamma = gi % gpc;
    const int sigma = gamma / g.nsg, sg = gamma % g.nsg;
    const int h = sigma & 1, u = sigma >> 1;
    const int a = l / g.w;
    const int v = (sg - a + g.nsg) % g.nsg;
    const int e = (u * g.nsg + v) * (g.q + 1) + comp;
    const size_t off = ((size_t)kc * g.n_rb + rb) * g.tile_bytes + g.plane_bytes + ((size_t)(e / 2) * 32 + 16 * h + l) * 4 + 2 * (e % 2);
    const uint16_t bits = *reinterpret_cast<const uint16_t*>(tiles + off);
    if (comp < g.q) scales[((size_t)n * Gn + gi) * g.q + comp] = bits;
    else offsets[(size_t)n * Gn + gi] = bits;
}

inline unsigned blocks_for(long long total, int threads) { return (unsigned)((total + threads - 1) / threads); }

}  // namespace

namespace {

template <int Q, int G>
int launch_pack_qg(const uint8_t* planes, const uint16_t* scales, const uint16_t* offsets, const Geo& g, uint8_t* packed, cudaStream_t stream) {
    const long long tiles = (long long)g.n_kc * g.n_rb, vectors = tiles * 2 * Q, words = tiles * g.gl * (Q + 1) / 2;
    if (vectors >= (1LL << 31) - 64 || words >= (1LL << 31) - 64) return (int)cudaErrorInvalidValue;
    Div by_rows;
    by_rows.set(g.n_rb);
    const unsigned plane_blocks = blocks_for(vectors, kPackWarps);
    pack_kernel<Q, G><<<plane_blocks + blocks_for(words, kPackWarps), 32 * kPackWarps, 0, stream>>>(
        planes, scales, offsets, packed, g, (int)plane_blocks, by_rows, (reinterpret_cast<uintptr_t>(planes) & 15) == 0);
    count_launch(1);
    return (int)cudaGetLastError();
}

template <int Q>
int launch_pack_q(const uint8_t* planes, const uint16_t* scales, const uint16_t* offsets, const Geo& g, uint8_t* packed, cudaStream_t stream) {
    switch (g.G) {
        case 32: return launch_pack_qg<Q, 32>(planes, scales, offsets, g, packed, stream);
        case 64: return launch_pack_qg<Q, 64>(planes, scales, offsets, g, packed, stream);
        default: return launch_pack_qg<Q, 128>(planes, scales, offsets, g, packed, stream);
    }
}

}  // namespace

int launch_pack(const uint8_t* planes, const __half* scales, const __half* offsets, const Geo& g,
                uint8_t* packed, cudaStream_t stream) {
    const uint16_t* s = reinterpret_cast<const uint16_t*>(scales);
    const uint16_t* z = reinterpret_cast<const uint16_t*>(offsets);
    switch (g.q) {
        case 1: return launch_pack_q<1>(planes, s, z, g, packed, stream);
        case 2: return launch_pack_q<2>(planes, s, z, g, packed, stream);
        case 3: return launch_pack_q<3>(planes, s, z, g, packed, stream);
        default: return launch_pack_q<4>(planes, s, z, g, packed, stream);
    }
}

int launch_unpack(const uint8_t* packed, const Geo& g, uint8_t* planes, __half* scales, __half* offsets,
                  cudaStream_t stream) {
    const uint8_t* tiles = packed + ELUTQ_HEADER_BYTES;
    const long long nb = (long long)g.q * g.N * (g.K / 8);
    unpack_planes_kernel<<<blocks_for(nb, 256), 256, 0, stream>>>(tiles, planes, g);
    const long long np = (long long)g.N * (g.K / g.G) * (g.q + 1);
    unpack_params_kernel<<<blocks_for(np, 256), 256, 0, stream>>>(
        tiles, reinterpret_cast<uint16_t*>(scales), reinterpret_cast<uint16_t*>(offsets), g);
    count_launch(2);
    return (int)cudaGetLastError();
}

}  // namespace elutq
