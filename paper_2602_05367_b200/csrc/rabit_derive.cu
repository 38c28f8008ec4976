// Writing a layer's packed image on the device: from a full-precision weight (derivation of the sign planes, fused with
// packing) or from canonical sign planes.
//
//   R_0 = W,   B_k = sign(R_{k-1}),   R_k = R_{k-1} - g_k (.) B_k (.) h_k        (Section 4.2, steps 1-3; Algorithm 2)
//
// The derivation is the step just before the inference hot path: at the end of training the sign matrices are derived once
// from the shared full-precision weight and frozen (end of Section 4.2).  Every weight entry is independent, so the kernel
// streams W once (4 bytes per weight in, 2K bits out) and writes both arrangements of the device layout directly.
// Arithmetic is fp32: the product g*h of two fp16 values is exact in fp32, so each residual update is one fp32 rounding;
// sign(0) = +1 (bit 0).
#include <cuda_fp16.h>

#include <cstring>

#include "rabit_internal.h"

namespace {

constexpr int kWarps = 8;
static_assert(kWarps * RABIT_TILE_COLS == RABIT_LUT_COLS, "one warp per column tile of a slice");

// What a layer's image needs besides the signs: the exchange buffer of all-ones words, zeroed flags and the header, which
// arrives as a kernel parameter (one host-to-device copy fewer).  Shared out over the CTAs of a kernel that writes signs.
struct HeaderWords {
    uint4 v[RABIT_HEADER_BYTES / 16];
};
struct Fills {
    uint4 *ones, *zero, *header_dst;
    size_t n_ones, n_zero;                                // 16-byte units
    HeaderWords header;
};
__device__ __forceinline__ void do_fills(const Fills& F) {
    if (blockIdx.x == 0 && threadIdx.x < RABIT_HEADER_BYTES / 16) F.header_dst[threadIdx.x] = F.header.v[threadIdx.x];
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < F.n_ones; i += (size_t)gridDim.x * blockDim.x)
        F.ones[i] = make_uint4(0xFFFFFFFFu, 0xFFFFFFFFu, 0xFFFFFFFFu, 0xFFFFFFFFu);
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < F.n_zero; i += (size_t)gridDim.x * blockDim.x)
        F.zero[i] = make_uint4(0u, 0u, 0u, 0u);
}

// Byte offset inside the look-up blocks of a row tile and slice (four row blocks, K KB each) of the byte that holds byte
// group `group` (0..31) of row `rl` (0..127) in path k.
__device__ __forceinline__ int slice_byte(int K, int k, int rl, int group) {
    const int l = rl & 31, s = (group - l) & 31;
    return ((rl >> 5) * K + k) * RABIT_LUT_PART_BYTES + (s >> 4) * 512 + l * 16 + (s & 15);
}

// One CTA per (row tile, slice of 256 columns), one warp per column tile; lane (gq, tq) owns rows 16p + gq + 8 alo and columns
// 16 ah + 4 tq + c, which are the 16 bytes per path it owns in the sign tile.  The sign bit of a residual is shifted into two words
// with one funnel shift each: in (c, p) order it is the tile's word (byte c, bit p), in (p, c) order a row's nibble, of which
// two neighbouring lanes make a byte of the look-up blocks.  Bound: latency.  11008 x 4096 at K = 2 takes 47 to 48 us for a floor
// of 32: 13.7 instructions per weight (loads, recurrence, both arrangements), issue slots 39 % and HBM 47 % busy, 15 warps per
// SM mostly waiting for W, of which 128 registers a thread leave no more than a part ahead.
// (Before: 43.9 us with a compare, a select and an OR per path and element, and 17 for a second kernel that gathered the
// look-up blocks from the tiles.)
template <int K>
__global__ void __launch_bounds__(kWarps * 32, 2)
rabit_derive_kernel(RabitGeom G, const float* __restrict__ W, const __half* __restrict__ g, const __half* __restrict__ h,
                    uint4* __restrict__ tiles, uint4* __restrict__ lut, const __grid_constant__ Fills F) {
    __shared__ __align__(16) unsigned char bytes[4 * K * RABIT_LUT_PART_BYTES];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int rt = blockIdx.x / G.n_cs, cs = blockIdx.x - rt * G.n_cs, ct = cs * kWarps + warp;
    const int gq = lane >> 2, tq = lane & 3;
    const bool inside = ct < G.n_ct;

    // W in four parts of 8 x 16 bytes, the next one in flight while the current one is worked through
    float4 w[2][8];
    auto load = [&](int part, float4 (&dst)[8]) {
        const int alo = part >> 1, ah = part & 1;
#pragma unroll
        for (int p = 0; p < 8; ++p) {
            const int row = rt * RABIT_TILE_ROWS + 16 * p + gq + 8 * alo;
            dst[p] = make_float4(0.f, 0.f, 0.f, 0.f);     // padded rows and columns: +1 signs
            if (inside && row < G.M) dst[p] = __ldcs(reinterpret_cast<const float4*>(W + (size_t)row * G.N + ct * RABIT_TILE_COLS + 16 * ah + 4 * tq));
        }
    };
    load(0, w[0]);
    do_fills(F);
    uint32_t out[K][4];
#pragma unroll
    for (int part = 0; part < 4; ++part) {
        if (part < 3) load(part + 1, w[(part + 1) & 1]);
        const int alo = part >> 1, ah = part & 1;
        float r[8][4];
#pragma unroll
        for (int p = 0; p < 8; ++p) {                     // (+ 0: a weight of -0 is +0, a NaN the positive one: bit 0)
            const float4 v = w[part & 1][p];
            r[p][0] = v.x + 0.f; r[p][1] = v.y + 0.f; r[p][2] = v.z + 0.f; r[p][3] = v.w + 0.f;
        }
#pragma unroll
        for (int k = 0; k < K; ++k) {
            uint32_t tile = 0u, nibbles = 0u;
#pragma unroll
            for (int c = 3; c >= 0; --c)
#pragma unroll
                for (int p = 7; p >= 0; --p) tile = __funnelshift_l(__float_as_uint(r[p][c]), tile, 1);
#pragma unroll
            for (int p = 7; p >= 0; --p)
#pragma unroll
                for (int c = 3; c >= 0; --c) nibbles = __funnelshift_l(__float_as_uint(r[p][c]), nibbles, 1);
            out[k][alo | (ah << 1)] = tile;
            if (k + 1 < K) {
                float hv[4] = {0.f, 0.f, 0.f, 0.f};
                if (inside) {
                    const uint2 raw = *reinterpret_cast<const uint2*>(h + (size_t)k * G.N + ct * RABIT_TILE_COLS + 16 * ah + 4 * tq);
                    const float2 a = __half22float2(*reinterpret_cast<const __half2*>(&raw.x)), b = __half22float2(*reinterpret_cast<const __half2*>(&raw.y));
                    hv[0] = a.x; hv[1] = a.y; hv[2] = b.x; hv[3] = b.y;
                }
#pragma unroll
                for (int p = 0; p < 8; ++p) {
                    const float gv = __half2float(g[(size_t)k * G.Mp + rt * RABIT_TILE_ROWS + 16 * p + gq + 8 * alo]);   // (zero in padded rows)
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        const float gb = __uint_as_float(__float_as_uint(gv) ^ (__float_as_uint(r[p][c]) & 0x80000000u));   // g * B, exact
                        r[p][c] = r[p][c] - gb * hv[c];   // the product is exact in fp32: one rounding
                    }
                }
            }
            // bytes of the look-up blocks: the even lane of a pair has columns 0..3 of the byte group, the odd one columns 4..7; the
            // even lane puts together the rows p = 0..3, the odd one p = 4..7
            const uint32_t other = __shfl_xor_sync(0xFFFFFFFFu, nibbles, 1);
            const int odd = tq & 1;
            uint32_t lo = ((odd ? other : nibbles) >> (16 * odd)) & 0xFFFFu, hi = ((odd ? nibbles : other) >> (16 * odd)) & 0xFFFFu;
            lo = (lo | (lo << 8)) & 0x00FF00FFu; lo = (lo | (lo << 4)) & 0x0F0F0F0Fu;
            hi = (hi | (hi << 8)) & 0x00FF00FFu; hi = (hi | (hi << 4)) & 0x0F0F0F0Fu;
            const uint32_t four = lo | (hi << 4);
#pragma unroll
            for (int i = 0; i < 4; ++i)
                bytes[slice_byte(K, k, 16 * (4 * odd + i) + gq + 8 * alo, 4 * warp + 2 * ah + (tq >> 1))] = (unsigned char)(four >> (8 * i));
        }
    }
    if (inside) {
#pragma unroll
        for (int k = 0; k < K; ++k) tiles[rabit_tile_pos(G, rt, k, ct) * 32 + lane] = make_uint4(out[k][0], out[k][1], out[k][2], out[k][3]);
    }
    __syncthreads();
    uint4* dst = lut + ((size_t)cs * G.n_rb + 4 * rt) * K * (RABIT_LUT_PART_BYTES / 16);
    for (int i = threadIdx.x; i < 4 * K * (RABIT_LUT_PART_BYTES / 16); i += kWarps * 32) dst[i] = reinterpret_cast<const uint4*>(bytes)[i];
}

// Canonical planes [K][M][N/32] -> look-up blocks: one warp per (slice, row block), lane = row.  A row's 32 bytes of the slice
// are its canonical bytes rotated left by the lane index.
__global__ void __launch_bounds__(kWarps * 32)
rabit_planes_to_lut_kernel(RabitGeom G, const uint32_t* __restrict__ planes, uint4* __restrict__ lut) {
    __shared__ uint32_t rows[kWarps][32][9];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const long long wid = (long long)blockIdx.x * kWarps + warp;
    if (wid >= (long long)G.n_cs * G.n_rb) return;
    const int cs = (int)(wid / G.n_rb), rb = (int)(wid - (long long)cs * G.n_rb), row = rb * RABIT_LUT_ROWS + lane, words = G.N / 32;
    for (int k = 0; k < G.K; ++k) {
        const uint32_t* src = planes + ((size_t)k * G.M + row) * words + cs * 8;
#pragma unroll
        for (int j = 0; j < 8; ++j) rows[warp][lane][j] = row < G.M && cs * 8 + j < words ? __ldcs(src + j) : 0u;
        uint32_t o[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const int at = j + (lane >> 2);
            o[j] = __byte_perm(rows[warp][lane][at & 7], rows[warp][lane][(at + 1) & 7], 0x3210u + 0x1111u * (lane & 3));
        }
        uint4* dst = lut + ((size_t)wid * G.K + k) * (RABIT_LUT_PART_BYTES / 16);
        dst[lane] = make_uint4(o[0], o[1], o[2], o[3]);
        dst[32 + lane] = make_uint4(o[4], o[5], o[6], o[7]);
    }
}

// Look-up blocks -> sign tiles: one CTA per (row tile, slice), one warp per column tile.  A tile word is eight rows of four
// columns: eight nibbles, each spread over the four bytes and shifted to its row block's bit.
__global__ void __launch_bounds__(kWarps * 32)
rabit_lut_to_tiles_kernel(RabitGeom G, const uint4* __restrict__ lut, uint4* __restrict__ tiles, const __grid_constant__ Fills F) {
    __shared__ __align__(16) unsigned char bytes[4 * RABIT_MAX_K * RABIT_LUT_PART_BYTES];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int rt = blockIdx.x / G.n_cs, cs = blockIdx.x - rt * G.n_cs, ct = cs * kWarps + warp;
    const int gq = lane >> 2, tq = lane & 3;
    do_fills(F);
    const uint4* src = lut + ((size_t)cs * G.n_rb + 4 * rt) * G.K * (RABIT_LUT_PART_BYTES / 16);
    for (int i = threadIdx.x; i < 4 * G.K * (RABIT_LUT_PART_BYTES / 16); i += kWarps * 32) reinterpret_cast<uint4*>(bytes)[i] = src[i];
    __syncthreads();
    if (ct >= G.n_ct) return;
    for (int k = 0; k < G.K; ++k) {
        uint32_t o[4];
#pragma unroll
        for (int a = 0; a < 4; ++a) {
            o[a] = 0u;
#pragma unroll
            for (int p = 0; p < 8; ++p) {
                const uint32_t n = (bytes[slice_byte(G.K, k, 16 * p + gq + 8 * (a & 1), 4 * warp + 2 * (a >> 1) + (tq >> 1))] >> (4 * (tq & 1))) & 0xFu;
                o[a] |= ((n * 0x00204081u) & 0x01010101u) << p;
            }
        }
        tiles[rabit_tile_pos(G, rt, k, ct) * 32 + lane] = make_uint4(o[0], o[1], o[2], o[3]);
    }
}

void make_fills(const RabitHeader& hdr, char* base, Fills* F) {
    static_assert(sizeof(RabitHeader) == RABIT_HEADER_BYTES, "the header travels as a kernel parameter");
    std::memcpy(&F->header, &hdr, sizeof(RabitHeader));
    F->header_dst = reinterpret_cast<uint4*>(base);
    F->ones = reinterpret_cast<uint4*>(base + hdr.off_partial);
    F->n_ones = (size_t)(hdr.off_flags - hdr.off_partial) / 16;
    F->zero = reinterpret_cast<uint4*>(base + hdr.off_flags);
    F->n_zero = (size_t)(hdr.off_lut - hdr.off_flags) / 16;
}

}  // namespace

// Both write the signs in both arrangements, the header and the resting state of the exchange buffer and the flags; the scales
// must be in place, the accumulate words are the caller's.
cudaError_t rabit_launch_derive(const RabitGeom& G, const RabitHeader& hdr, char* base, const float* W, cudaStream_t stream) {
    const long long blocks = (long long)G.n_rt * G.n_cs;
    if (blocks > 0x7FFFFFFFLL) return cudaErrorInvalidValue;
    Fills F;
    make_fills(hdr, base, &F);
    const __half *g = reinterpret_cast<const __half*>(base + hdr.off_g), *h = reinterpret_cast<const __half*>(base + hdr.off_h);
    uint4 *tiles = reinterpret_cast<uint4*>(base + hdr.off_bits), *lut = reinterpret_cast<uint4*>(base + hdr.off_lut);
    if (G.K == 1) rabit_derive_kernel<1><<<(unsigned int)blocks, kWarps * 32, 0, stream>>>(G, W, g, h, tiles, lut, F);
    else if (G.K == 2) rabit_derive_kernel<2><<<(unsigned int)blocks, kWarps * 32, 0, stream>>>(G, W, g, h, tiles, lut, F);
    else rabit_derive_kernel<3><<<(unsigned int)blocks, kWarps * 32, 0, stream>>>(G, W, g, h, tiles, lut, F);
    return cudaGetLastError();
}

// `planes` may lie in the section of the sign tiles: the look-up blocks are made from the planes, the tiles from the look-up blocks.
cudaError_t rabit_launch_pack_planes(const RabitGeom& G, const RabitHeader& hdr, char* base, const uint32_t* planes, cudaStream_t stream) {
    const long long blocks = (long long)G.n_rt * G.n_cs;
    if (blocks > 0x7FFFFFFFLL) return cudaErrorInvalidValue;
    Fills F;
    make_fills(hdr, base, &F);
    uint4 *tiles = reinterpret_cast<uint4*>(base + hdr.off_bits), *lut = reinterpret_cast<uint4*>(base + hdr.off_lut);
    rabit_planes_to_lut_kernel<<<(unsigned int)((blocks * 4 + kWarps - 1) / kWarps), kWarps * 32, 0, stream>>>(G, planes, lut);
    rabit_lut_to_tiles_kernel<<<(unsigned int)blocks, kWarps * 32, 0, stream>>>(G, lut, tiles, F);
    return cudaGetLastError();
}
