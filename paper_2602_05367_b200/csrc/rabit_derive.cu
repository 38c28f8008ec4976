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

#include <algorithm>
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

// 16 bytes global -> shared, asynchronous, not through L1 (valid false: zeros)
__device__ __forceinline__ void copy_async_16(uint32_t dst, const void* src, bool valid) {
    const uint32_t size = valid ? 16u : 0u;
    asm volatile("cp.async.cg.shared.global.L2::128B [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(size) : "memory");
}
template <int N>
__device__ __forceinline__ void copy_async_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// A persistent CTA takes (row tile, slice of 256 columns) blocks in turn, one warp per column tile; lane (gq, tq) owns rows 16p + gq + 8 alo and
// columns 16 ah + 4 tq + c, which are the 16 bytes per path it owns in the sign tile.  The sign bit of a residual is shifted into the
// tile's word (byte c, bit p) with one funnel shift; transposed, two neighbouring lanes' words are four bytes of the look-up blocks each.
// W comes in parts of 4 KB a warp (a quarter of its 128 x 32 weights) by asynchronous copies into a ring of three parts of its own in shared
// memory, two ahead of the one at hand and across block borders; a lane reads back what it copied itself, so no barrier is involved.
// The scales of the next block are fetched beside the work on this one.  Two CTAs per SM, which for three paths takes scales of one block only in
// shared memory (of two 48.6 us, one CTA per SM, instead of 42.6).  Bound: HBM with one path (11008 x 4096, 200 MB in and out: 32 us), beyond that the
// recurrence's instructions beside it; two paths 36.5 (47.9 with W in registers, at most a part ahead), 28672 x 8192 161 (256).
constexpr int kRingParts = 3;
constexpr int kPartBytes = 32 * 8 * 16;
template <int K>
struct DeriveSmem {
    static constexpr int kBytes = kWarps * kRingParts * kPartBytes;                          // behind the ring: the look-up bytes of a block
    static constexpr int kScales = kBytes + 4 * K * RABIT_LUT_PART_BYTES;                    // then g and h of the block, fp32
    static constexpr int kScaleFloats = (K - 1) * (RABIT_TILE_ROWS + RABIT_LUT_COLS);        // (the last path's are not needed)
    static constexpr int kTotal = kScales + kScaleFloats * 4;
    static_assert(2 * (kTotal + 1024) <= 228 * 1024, "two CTAs per SM");
};
template <int K>
__global__ void __launch_bounds__(kWarps * 32, 2)
rabit_derive_kernel(RabitGeom G, const float* __restrict__ W, const __half* __restrict__ g, const __half* __restrict__ h,
                    uint4* __restrict__ tiles, uint4* __restrict__ lut, uint32_t n_blocks, const __grid_constant__ Fills F) {
    using S = DeriveSmem<K>;
    extern __shared__ __align__(16) unsigned char smem[];
    unsigned char* bytes = smem + S::kBytes;
    float* scales = reinterpret_cast<float*>(smem + S::kScales);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int gq = lane >> 2, tq = lane & 3;
    const uint32_t ring = (uint32_t)__cvta_generic_to_shared(smem) + (uint32_t)(warp * kRingParts * kPartBytes + lane * 16);

    // part `part` of block b of W into ring slot `slot` (padded rows and columns, and blocks beyond the last: zeros, i.e. +1 signs)
    auto fetch = [&](uint32_t b, int part, int slot) {
        const int rt = (int)(b / (uint32_t)G.n_cs), ct = (int)(b - (uint32_t)rt * G.n_cs) * kWarps + warp, row0 = rt * RABIT_TILE_ROWS + gq + 8 * (part >> 1);
        const bool inside = b < n_blocks && ct < G.n_ct;
        const float* src = W + (size_t)row0 * G.N + ct * RABIT_TILE_COLS + 16 * (part & 1) + 4 * tq;
#pragma unroll
        for (int p = 0; p < 8; ++p) {
            const bool valid = inside && row0 + 16 * p < G.M;
            copy_async_16(ring + (uint32_t)(slot * kPartBytes + p * 512), valid ? src + (size_t)(16 * p) * G.N : W, valid);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    // output and input scales of block b, a few per thread
    constexpr int kPerThread = (S::kScaleFloats + kWarps * 32 - 1) / (kWarps * 32);
    __half next[kPerThread > 0 ? kPerThread : 1];
    auto fetch_scales = [&](uint32_t b) {
        const int rt = (int)(b / (uint32_t)G.n_cs), cs = (int)(b - (uint32_t)rt * G.n_cs);
#pragma unroll
        for (int u = 0; u < kPerThread; ++u) {
            const int i = threadIdx.x + u * kWarps * 32, k = i / (RABIT_TILE_ROWS + RABIT_LUT_COLS), j = i - k * (RABIT_TILE_ROWS + RABIT_LUT_COLS);
            const int col = cs * RABIT_LUT_COLS + j - RABIT_TILE_ROWS;
            next[u] = __half();
            if (i < S::kScaleFloats && b < n_blocks) {
                if (j < RABIT_TILE_ROWS) next[u] = g[(size_t)k * G.Mp + rt * RABIT_TILE_ROWS + j];       // (zero in padded rows)
                else if (col < G.N) next[u] = h[(size_t)k * G.N + col];
            }
        }
    };
    auto keep_scales = [&]() {
#pragma unroll
        for (int u = 0; u < kPerThread; ++u) {
            const int i = threadIdx.x + u * kWarps * 32;
            if (i < S::kScaleFloats) scales[i] = __half2float(next[u]);
        }
    };

    fetch(blockIdx.x, 0, 0);
    fetch(blockIdx.x, 1, 1);
    fetch_scales(blockIdx.x);
    do_fills(F);
    keep_scales();
    __syncthreads();
    const uint32_t own_half = tq & 1 ? 0xF0F0F0F0u : 0x0F0F0F0Fu;
    const int turn = tq & 1 ? 28 : 4;
    int slot = 0, ahead = 2;                              // ring slots of the part at hand and of the one to fetch
    for (uint32_t b = blockIdx.x; b < n_blocks; b += gridDim.x) {
        const int rt = (int)(b / (uint32_t)G.n_cs), cs = (int)(b - (uint32_t)rt * G.n_cs), ct = cs * kWarps + warp;
        const bool inside = ct < G.n_ct;
        fetch_scales(b + gridDim.x);
        uint32_t out[K][4];
#pragma unroll
        for (int part = 0; part < 4; ++part) {
            fetch(part < 2 ? b : b + gridDim.x, (part + 2) & 3, ahead);     // (into the slot of the part before this one)
            ahead = ahead == kRingParts - 1 ? 0 : ahead + 1;
            copy_async_wait<2>();
            const int alo = part >> 1, ah = part & 1;
            float r[8][4];
#pragma unroll
            for (int p = 0; p < 8; ++p) {                 // (+ 0: a weight of -0 is +0, a NaN the positive one: bit 0)
                float4 v;
                asm volatile("ld.shared.v4.f32 {%0,%1,%2,%3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(ring + (uint32_t)(slot * kPartBytes + p * 512)) : "memory");
                r[p][0] = v.x + 0.f; r[p][1] = v.y + 0.f; r[p][2] = v.z + 0.f; r[p][3] = v.w + 0.f;
            }
            slot = slot == kRingParts - 1 ? 0 : slot + 1;
#pragma unroll
            for (int k = 0; k < K; ++k) {
                uint32_t tile = 0u;
#pragma unroll
                for (int c = 3; c >= 0; --c)
#pragma unroll
                    for (int p = 7; p >= 0; --p) tile = __funnelshift_l(__float_as_uint(r[p][c]), tile, 1);
                out[k][alo | (ah << 1)] = tile;
                if (k + 1 < K) {
                    const float* gk = scales + k * (RABIT_TILE_ROWS + RABIT_LUT_COLS);
                    const float4 hv = *reinterpret_cast<const float4*>(gk + RABIT_TILE_ROWS + warp * RABIT_TILE_COLS + 16 * ah + 4 * tq);
                    const float hc[4] = {hv.x, hv.y, hv.z, hv.w};
#pragma unroll
                    for (int p = 0; p < 8; ++p) {
                        const float gv = gk[16 * p + gq + 8 * alo];
#pragma unroll
                        for (int c = 0; c < 4; ++c) {
                            const float gb = __uint_as_float(__float_as_uint(gv) ^ (__float_as_uint(r[p][c]) & 0x80000000u));   // g * B, exact
                            r[p][c] = r[p][c] - gb * hc[c];   // the product is exact in fp32: one rounding
                        }
                    }
                }
                // Bytes of the look-up blocks.  The word has bit p of byte c; with the two halves of its bytes transposed as 4 x 4 bit matrices byte i
                // holds the columns of row block i in its low half, those of row block 4 + i in its high half.  The even lane of a pair has columns
                // 0..3 of the byte group, the odd one columns 4..7; the even lane puts together the rows p = 0..3, the odd one p = 4..7.
                uint32_t rows = tile, t = (rows ^ (rows >> 7)) & 0x00AA00AAu;
                rows ^= t ^ (t << 7);
                t = (rows ^ (rows >> 14)) & 0x0000CCCCu;
                rows ^= t ^ (t << 14);
                const uint32_t other = __shfl_xor_sync(0xFFFFFFFFu, rows, 1);
                const uint32_t four = (rows & own_half) | (__funnelshift_l(other, other, turn) & ~own_half);
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    bytes[slice_byte(K, k, 16 * (4 * (tq & 1) + i) + gq + 8 * alo, 4 * warp + 2 * ah + (tq >> 1))] = (unsigned char)(four >> (8 * i));
            }
        }
        if (inside) {
#pragma unroll
            for (int k = 0; k < K; ++k) tiles[rabit_tile_pos(G, rt, k, ct) * 32 + lane] = make_uint4(out[k][0], out[k][1], out[k][2], out[k][3]);
        }
        __syncthreads();
        keep_scales();                                    // (nobody reads this block's any more)
        uint4* dst = lut + ((size_t)cs * G.n_rb + 4 * rt) * K * (RABIT_LUT_PART_BYTES / 16);
        for (int i = threadIdx.x; i < 4 * K * (RABIT_LUT_PART_BYTES / 16); i += kWarps * 32) dst[i] = reinterpret_cast<const uint4*>(bytes)[i];
        __syncthreads();
    }
    copy_async_wait<0>();
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

template <int K>
cudaError_t launch_derive(const RabitGeom& G, const float* W, const __half* g, const __half* h, uint4* tiles, uint4* lut, uint32_t blocks, unsigned int grid, int device,
                          const Fills& F, cudaStream_t stream) {
    static bool done[64] = {};                            // function attributes are per device
    if (device < 0 || device >= 64 || !done[device]) {
        cudaError_t e = cudaFuncSetAttribute(rabit_derive_kernel<K>, cudaFuncAttributeMaxDynamicSharedMemorySize, DeriveSmem<K>::kTotal);
        if (e != cudaSuccess) return e;
        if (device >= 0 && device < 64) done[device] = true;
    }
    rabit_derive_kernel<K><<<grid, kWarps * 32, DeriveSmem<K>::kTotal, stream>>>(G, W, g, h, tiles, lut, blocks, F);
    return cudaGetLastError();
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
    int device = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&device);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device);
    if (e != cudaSuccess) return e;
    const unsigned int grid = (unsigned int)std::min<long long>(blocks, 2LL * sms);
    return G.K == 1 ? launch_derive<1>(G, W, g, h, tiles, lut, (uint32_t)blocks, grid, device, F, stream)
         : G.K == 2 ? launch_derive<2>(G, W, g, h, tiles, lut, (uint32_t)blocks, grid, device, F, stream)
                    : launch_derive<3>(G, W, g, h, tiles, lut, (uint32_t)blocks, grid, device, F, stream);
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
