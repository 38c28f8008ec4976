// Decode GEMV for 3..8 batch rows: the batch sits in the N dimension of an f16 tensor-core MMA.
//
//   y[b][i] = sum_k g_k[i] * sum_j (B_k[i][j] h_k[j]) * x[b][j]                              (Section 4.1, Eq. 2)
//
// The table-driven kernel (rabit_gemv_lut.cu) pays per batch row; the integer tensor-core GEMV spends four of an MMA's
// eight columns per batch row and needs a pass over x first.  Here the A operand of mma.sync.m16n8k16 is +-h_k expanded in
// registers from the sign tiles (the weight bit flips the sign bit of the fp16 input scale: exact), B is x as it is, the
// accumulators are fp32: products are exact, 8 batch rows per MMA, no digits, no scale search.  The cost is that of the
// expansion and does not depend on the batch.
//
// Expansion.  Shifts, byte permutes, multiplications and logic instructions each take two issue clocks of an SM
// sub-partition, and issue slots, not the tensor pipe, bound this kernel.  The two weight bits of an A register (two fp16 values)
// must be 16 apart in the word, i.e. two columns apart.  A multiplication by a power of two (a kernel parameter, so that the
// compiler keeps it one) brings those of an odd row block to bits 15 and 31: one logic instruction, (v & 0x80008000) ^ h.
// The even row block below then has its bits at 14 and 30, where a bit alone is the fp16 number 2: an AND and one half2 fused
// multiply-add, h - 2 h or h - 0 h (exact; one issue clock), without a shift of its own.
//
// Operand mapping.  A sign tile (rabit_layout.h) gives lane (gq, tq) four words w[a]; byte c of word a has in bit p the
// sign of row 16p + gq + 8(a & 1), column 16(a >> 1) + 4tq + c of the tile.  For the k-step kh = a >> 1 (16 columns) and
// the row block p, the MMA's k slots (2tq, 2tq+1, 2tq+8, 2tq+9) of lane (gq, tq) are taken to be the tile columns
// 16kh + 4tq + (0, 2, 1, 3): any fixed assignment of slots to columns is valid as long as A and B use the same one.  Then
//     a0 = +-h(cols 0,2) for row gq      from bits p, 16+p of w[2kh] * 2^(15-p)      a1 = the same, row gq + 8, from w[2kh+1]
//     a2 = +-h(cols 1,3) for row gq      from bits 8+p, 24+p of w[2kh] * 2^(7-p)     a3 = row gq + 8, from w[2kh+1]
//     b0 = x[n = gq][cols 0,2]           b1 = x[n = gq][cols 1,3]         (one 8-byte load per lane and k-step, two permutes)
// and the accumulator lane holds rows gq, gq + 8 of the block and batch rows 2tq, 2tq + 1.
//
// Work split.  The launch's layers are n_rt row tiles x n_cs slices of 256 columns each; the host cuts these pairs, in that
// order, into contiguous ranges, one per SM, worked through by one group of 16 warps or cut once more for two groups of 8
// (struct Planner).  The part of a range inside one row tile is a segment.  Warp w of a group works on path w % K and shares the column tiles of the segment
// with the other warps of that path.  A warp streams its tiles through a ring of its own in shared memory with asynchronous
// 16-byte copies (one per lane and tile, each lane reads back only what it copied itself, so no barrier is involved),
// kRing - 1 tiles ahead: with 16 warps per SM that keeps about 56 KB per SM in flight, which is what the HBM latency needs
// (with the tiles prefetched into registers, two to four per warp, the kernel ran at the speed of its memory latency, 1.1
// to 1.7 TB/s).  At the end of a segment every warp writes its accumulators to its own slot of shared memory and the group adds
// the slots path by path in a fixed order (deterministic), applying g_k to each path's sum.  A segment that is a whole row
// tile stores y.  Otherwise every output goes, as in the table-driven kernel, into the row's 64-bit accumulate word with one
// integer atomic (fixed-point grid of the packer, arrival count in bits 55..62, bit 63 = non-finite); the thread whose add
// completes a row (the count reaches the number of segments of that row tile) rounds it to fp16, stores y and clears the
// word.  A contribution that covers s slices is shifted by s * 2^fix_bits, so the total shift is the same n_cs * 2^fix_bits
// for every split.  Nothing waits for another CTA.
//
// What bounds it (B200, clocks per 512-byte tile and SM): about 70 in the steady state, of which the loads of x and h are 10 %;
// the rest is 16 MMAs of about 2 clocks and the expansion, which hardly overlap.  Segment ends are what a split can save: an
// arrival count found by searching a table of range bounds in constant memory, cold in every launch, cost 1 us at each (it
// now comes with the range).  4096 x 14336 at 5 rows 13.1 -> 11.3 us, 4096 x 4096 at 8 7.1 -> 5.9, 28672 x 8192 at 8 37.9 -> 37.6.
#include <cuda_fp16.h>

#include <algorithm>
#include <cstring>
#include <vector>

#include "rabit_internal.h"

namespace {

constexpr int kThreads = 512;
constexpr int kRows = 8;                               // batch rows of a pass: an MMA's columns
constexpr int kRing = 8;                               // sign tiles a warp keeps in flight or in use (a power of two)
constexpr int kMaxRanges = 320;                       // two per SM of the largest device
constexpr long long kMaxPairs = 1LL << 23;
constexpr int kMaxGroup = 8;
constexpr int kSlotStride = 128 + 4;                  // floats per batch row of a slot: the pad spreads a warp's store over all banks
constexpr unsigned long long kSumMask = (1ULL << 55) - 1;

// Cost model (B200): a sign tile takes the SM about 70 clocks (8 % more when three paths are dealt to 8 warps); a segment end
// inside a range costs one group of 16 warps 2 us, one of two groups less than half (the other works on); a group whose partner is idle
// runs at 1 / kAlone of the time; publishing parts of row tiles takes 0.6 us and 128 * batch words per part at 80 words per clock over the GPU.
constexpr double kTileClocks = 70.0, kUneven3 = 1.08, kSegmentUs1 = 2.0, kSegmentUs2 = 0.75, kAlone = 1.4, kPublishUs = 0.6;

struct F16Layer {
    const uint4* tiles;
    const __half* g;
    const __half* h;
    const __half* x;
    __half* y;
    unsigned long long* acc;        // [16][Mp], all zero between calls
    unsigned int* status;           // RABIT_CHECKED builds: set to 2 when an index check fails (the access is skipped)
    int M, N, Mp, n_rt, n_ct, n_cs;
    int fix_bits;
    float inv_unit, unit, limit;
};
// A group's range of the launch's (row tile, slice) pairs, counted over its layers, and how many ranges touch the row tile at
// its start and at its end (those between are its own).
struct F16Range {
    int start;
    unsigned char first, last;
    unsigned short pad_;
};
struct F16Params {
    int n_layers, K, batch;
    uint32_t four, two_pow_8;       // 4 and 256: multipliers the compiler cannot fold into shifts
    int pair0[kMaxGroup];           // pairs of the layers before each
    F16Layer layer[kMaxGroup];
    F16Range range[kMaxRanges + 1]; // of group q of CTA c: range[GROUPS * c + q], up to the start of the next
};

// Checked build (-DRABIT_CHECKED, python paper_2602_05367_b200/build.py --checked): every index that addresses global or
// shared memory is compared with its range first; a violation is recorded in the layer's status word and the access is
// skipped (nothing traps).  In the ordinary build the checks compile to nothing.
#ifdef RABIT_CHECKED
#define RABIT_IN_RANGE(cond) ((cond) ? true : (atomicExch(P.layer[0].status, 2u), false))
#else
#define RABIT_IN_RANGE(cond) true
#endif

__device__ __forceinline__ uint32_t prmt(uint32_t a, uint32_t b, uint32_t s) {
    uint32_t r;
    asm("prmt.b32 %0, %1, %2, %3;" : "=r"(r) : "r"(a), "r"(b), "r"(s));
    return r;
}
// (a & 0x80008000) ^ c: the sign bits of two fp16 values, applied to a pair of input scales
__device__ __forceinline__ uint32_t flip(uint32_t a, uint32_t c) {
    uint32_t r;
    asm volatile("lop3.b32 %0, %1, 0x80008000, %2, 0x6A;" : "=r"(r) : "r"(a), "r"(c));
    return r;
}
// The same with the sign bits at 14 and 30: bit 14 alone is the fp16 number 2, so h - 2 h or h - 0 h, exact.
__device__ __forceinline__ uint32_t flip_below(uint32_t a, __half2 minus_h, uint32_t h) {
    const uint32_t two = a & 0x40004000u;
    const __half2 r = __hfma2(*reinterpret_cast<const __half2*>(&two), minus_h, *reinterpret_cast<const __half2*>(&h));
    return *reinterpret_cast<const uint32_t*>(&r);
}
// barrier of one group of warps (ids 1 and 2; 0 is left to __syncthreads)
template <int kGroupThreads>
__device__ __forceinline__ void group_sync(int group) {
    asm volatile("bar.sync %0, %1;" ::"r"(group + 1), "n"(kGroupThreads) : "memory");
}
// a * m on the multiply-add pipe (m is a power of two the compiler does not know)
__device__ __forceinline__ uint32_t mul_lo(uint32_t a, uint32_t m) {
    uint32_t r;
    asm volatile("mul.lo.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(m));
    return r;
}
__device__ __forceinline__ void mma_f16(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
                 : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
// 16 bytes global -> shared, asynchronous, not through L1; one group per call so that groups and tiles count alike
__device__ __forceinline__ void copy_async_16(uint32_t dst_smem, const void* src, bool valid) {
    if (valid) asm volatile("cp.async.cg.shared.global.L2::128B [%0], [%1], 16;" ::"r"(dst_smem), "l"(src) : "memory");
    asm volatile("cp.async.commit_group;" ::: "memory");
}
template <int N>
__device__ __forceinline__ void copy_async_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}
__device__ __forceinline__ uint4 lds_128(uint32_t addr) {
    uint4 v;
    asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr) : "memory");
    return v;
}

// One output of a segment from the warps' slots: warp w holds path w % KK; the paths' sums are formed warp by warp in the
// order of the warps and scaled by the path's output scale.
template <int KK, int kWarps>
__device__ __forceinline__ float path_sums(const float* col, const __half (&g)[RABIT_MAX_K]) {
    float sk[KK];
#pragma unroll
    for (int kk = 0; kk < KK; ++kk) sk[kk] = 0.f;
#pragma unroll
    for (int wv = 0; wv < kWarps; ++wv) sk[wv % KK] += col[(size_t)wv * (kRows * kSlotStride)];
    float v = 0.f;
#pragma unroll
    for (int kk = 0; kk < KK; ++kk) v = fmaf(__half2float(g[kk]), sk[kk], v);
    return v;
}

// GROUPS = 1: the CTA's 16 warps work on one range of pairs; 2: two groups of 8 on a range each, sharing nothing but the SM.
template <int GROUPS>
__global__ void __launch_bounds__(kThreads, 1)
rabit_gemv_f16_kernel(const __grid_constant__ F16Params P) {
    constexpr int kWarps = kThreads / 32 / GROUPS, kGroupThreads = kWarps * 32;
    constexpr int kGroupFloats = kWarps * kRows * kSlotStride + kWarps * kRing * 128;
    extern __shared__ __align__(16) float smem_f[];                      // per group: [kWarps][kRows][kSlotStride] partial outputs, then the warps' rings
    const int group = GROUPS == 1 ? 0 : threadIdx.x / kGroupThreads;
    const int tid = threadIdx.x % kGroupThreads, lane = tid & 31, warp = tid >> 5;
    const int gq = lane >> 2, tq = lane & 3;
    float* slots = smem_f + (size_t)group * kGroupFloats;
    // the lane's 16 bytes of ring slot 0 of its warp; slot r is r * 512 bytes further
    const uint32_t ring = (uint32_t)__cvta_generic_to_shared(slots) + (uint32_t)(kWarps * kRows * kSlotStride * sizeof(float)) +
                          (uint32_t)((warp * kRing * 32 + lane) * 16);

    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    bool waited = false;
    const int worker = GROUPS * (int)blockIdx.x + group;
    // The launch parameters sit in constant memory, cold in every launch (a first touch is a trip to L2): the layers' lines are
    // touched here, a warp each, while the others read the range.
    if (warp > 0 && (warp - 1) * 64 < P.n_layers * (int)sizeof(F16Layer)) {
        const uint32_t word = reinterpret_cast<const uint32_t*>(P.layer)[(warp - 1) * 16];
        asm volatile("" ::"r"(word));
    }
    const F16Range range = P.range[worker];
    int u = range.start, l = 0;
    const int u_first = u, u_end = P.range[worker + 1].start;
    while (l + 1 < P.n_layers && u >= P.pair0[l + 1]) ++l;

    // every warp works on ONE path: path k = warp % K, and the column tiles of a segment are dealt out among the
    // group's warps of that path (16 warps and K = 3: six, five and five)
    const int k = warp % P.K;
    const int n_same = (kWarps - k + P.K - 1) / P.K, j0 = warp / P.K;

    // A segment: row tile rt, column tiles [ct0, c1) of which this warp takes every n_same-th, starting at ct0.
    struct Segment {
        int l, rt, n_slices, arrivals, ct0, n_my;
        const uint4* wsrc;                                               // the warp's first tile (this lane's 16 bytes)
    };
    auto next_segment = [&]() {                                          // the segment that starts at pair u; advances u
        const F16Layer& L = P.layer[l];
        const int in_layer = u - P.pair0[l], n_cs = L.n_cs, n_ct = L.n_ct;
        Segment sg;
        sg.l = l;
        sg.rt = in_layer / n_cs;
        const int s0 = in_layer - sg.rt * n_cs, s1 = min(n_cs, s0 + (u_end - u));
        sg.n_slices = s1 - s0;
        sg.arrivals = sg.n_slices == n_cs ? 1 : u == u_first ? range.first : range.last;
        u += sg.n_slices;
        const int c1 = min(n_ct, s1 * 8);                              // a slice is eight column tiles
        sg.ct0 = s0 * 8 + j0;
        sg.n_my = sg.ct0 < c1 ? (c1 - sg.ct0 + n_same - 1) / n_same : 0;
        sg.wsrc = L.tiles + (size_t)(sg.rt * P.K + k) * n_ct * 32 + sg.ct0 * 32 + lane;
        if (s1 == n_cs && sg.rt + 1 == L.n_rt) ++l;
        return sg;
    };
    auto prefill = [&](const Segment& sg) {                              // the first kRing - 1 tiles of the warp; weights never depend on the stream's past
        [[maybe_unused]] const F16Layer& L = P.layer[sg.l];
#pragma unroll
        for (int i = 0; i < kRing - 1; ++i)
            copy_async_16(ring + i * 512, sg.wsrc + (size_t)i * n_same * 32,
                          i < sg.n_my && RABIT_IN_RANGE(sg.wsrc + (size_t)i * n_same * 32 >= L.tiles &&
                                                        sg.wsrc + (size_t)i * n_same * 32 < L.tiles + (size_t)L.n_rt * P.K * L.n_ct * 32));
    };
    bool more = u < u_end;
    Segment sg;
    if (more) {
        sg = next_segment();
        prefill(sg);
    }
    while (more) {
        const F16Layer& L = P.layer[sg.l];
        const int rt = sg.rt, ct0 = sg.ct0, n_my = sg.n_my, n_ct = L.n_ct;
        const __half *const h_base = L.h, *const x_base = L.x;
        const int hk = k * L.N + 4 * tq;                                  // element offsets (K * N and 8 * N fit 31 bits: N <= 65280)
        const int xb = min(gq, P.batch - 1) * L.N + 4 * tq;               // lanes beyond the batch read its last row; their columns are never stored
        const uint4* wsrc = sg.wsrc;
        float acc[8][4];
#pragma unroll
        for (int p = 0; p < 8; ++p)
#pragma unroll
            for (int e = 0; e < 4; ++e) acc[p][e] = 0.f;

        // input scales and activations of the lane's four columns of k-step kh of column tile ct, as loaded (columns 0,1 | 2,3)
        auto fetch_hx = [&](int ct, int kh, uint2& fh, uint2& fx) {
            const int off = ct * 32 + 16 * kh;
            if (!RABIT_IN_RANGE(off >= 0 && hk + off + 4 <= P.K * L.N)) return;
            fh = __ldg(reinterpret_cast<const uint2*>(h_base + hk + off));
            if (RABIT_IN_RANGE(xb + off + 4 <= P.batch * L.N)) fx = __ldcg(reinterpret_cast<const uint2*>(x_base + xb + off));
        };

        __half gk[RABIT_MAX_K];                                           // output scales of the thread's row (the same row for all its outputs), loaded long before they are used
#pragma unroll
        for (int kk = 0; kk < RABIT_MAX_K; ++kk)
            gk[kk] = kk < P.K && RABIT_IN_RANGE(rt >= 0 && rt < L.n_rt) ? L.g[(size_t)kk * L.Mp + rt * RABIT_TILE_ROWS + (tid & 127)] : __half();
        // weights kRing - 1 tiles ahead (HBM latency), scales and activations one tile ahead, k-step by k-step in place
        if (!waited) {
            asm volatile("griddepcontrol.wait;" ::: "memory");            // x, y and the accumulate words only after this
            waited = true;
        }
        uint2 fh[2], fx[2];
#pragma unroll
        for (int kh = 0; kh < 2; ++kh) fetch_hx(min(ct0, n_ct - 1), kh, fh[kh], fx[kh]);
        for (int i = 0; i < n_my; ++i) {
            {
                const int ct = ct0 + i * n_same;
                const int ia = i + kRing - 1;                            // the tile that takes the slot freed in the last round
                copy_async_16(ring + (ia & (kRing - 1)) * 512, wsrc + (size_t)ia * n_same * 32,
                              ia < n_my && RABIT_IN_RANGE(wsrc + (size_t)ia * n_same * 32 >= L.tiles &&
                                                          wsrc + (size_t)ia * n_same * 32 < L.tiles + (size_t)L.n_rt * P.K * n_ct * 32));
                copy_async_wait<kRing - 1>();                            // tile i has landed (one group per tile, also for the tiles that do not exist)
                const uint4 wv = lds_128(ring + (i & (kRing - 1)) * 512);
                const int ct_next = min(ct + n_same, n_ct - 1);        // beyond the segment: a valid address, never used
                const uint32_t w[4] = {wv.x, wv.y, wv.z, wv.w};
#pragma unroll
                for (int kh = 0; kh < 2; ++kh) {
                    const uint32_t h02 = prmt(fh[kh].x, fh[kh].y, 0x5410), h13 = prmt(fh[kh].x, fh[kh].y, 0x7632);
                    const uint32_t b0 = prmt(fx[kh].x, fx[kh].y, 0x5410), b1 = prmt(fx[kh].x, fx[kh].y, 0x7632);
                    const __half2 m02 = __hneg2(*reinterpret_cast<const __half2*>(&h02)), m13 = __hneg2(*reinterpret_cast<const __half2*>(&h13));
                    fetch_hx(ct_next, kh, fh[kh], fx[kh]);                // the same k-step of the warp's next tile, in place
                    // u = w * 2^(7-p): bit p of bytes 1 and 3 -> bits 15 and 31, bit p - 1 one below;  v = u * 2^8: the same for bytes 0 and 2
                    uint32_t ul = w[2 * kh], uh = w[2 * kh + 1];
                    uint32_t vl = mul_lo(ul, P.two_pow_8), vh = mul_lo(uh, P.two_pow_8);
#pragma unroll
                    for (int p = 7; p > 0; p -= 2) {
                        mma_f16(acc[p], flip(vl, h02), flip(vh, h02), flip(ul, h13), flip(uh, h13), b0, b1);
                        mma_f16(acc[p - 1], flip_below(vl, m02, h02), flip_below(vh, m02, h02), flip_below(ul, m13, h13), flip_below(uh, m13, h13), b0, b1);
                        if (p > 1) {
                            ul = mul_lo(ul, P.four); uh = mul_lo(uh, P.four);
                            vl = mul_lo(vl, P.four); vh = mul_lo(vh, P.four);
                        }
                    }
                }
            }
        }
        copy_async_wait<0>();
        // the next segment's first tiles set off now: they cross HBM while this segment is added up
        const int n_slices = sg.n_slices, arrivals = sg.arrivals;
        more = u < u_end;
        if (more) {
            sg = next_segment();
            prefill(sg);
        }
        constexpr int kPer = kRows * 128 / kGroupThreads;                     // outputs per thread (2 or 4)
        // ---- the warp's partial outputs -> its slot; slot layout [batch row][row of the tile]
        float* mine = slots + (size_t)warp * (kRows * kSlotStride);
        const bool slot_ok = RABIT_IN_RANGE(mine + (kRows - 1) * kSlotStride + 127 < smem_f + GROUPS * kGroupFloats);
#pragma unroll
        for (int p = 0; p < 8; ++p) {
            if (!slot_ok) break;
            const int b = 2 * tq, row = 16 * p + gq;
            mine[(b) * kSlotStride + row] = acc[p][0];
            mine[(b + 1) * kSlotStride + row] = acc[p][1];
            mine[(b) * kSlotStride + row + 8] = acc[p][2];
            mine[(b + 1) * kSlotStride + row + 8] = acc[p][3];
        }
        group_sync<kGroupThreads>(group);
        // ---- fixed-order sum over the warps, then one atomic per output of the segment
        // (thread t owns row t & 127 of the tile and the batch rows (t >> 7) + 4 i; rows beyond the batch are computed from
        // whatever their MMA columns held and dropped)
        unsigned long long old[kPer], add[kPer];
        bool bad[kPer];
#pragma unroll
        for (int i = 0; i < kPer; ++i) {
            const int o = tid + i * kGroupThreads, b = o >> 7, rl = o & 127;
            // sum_k g_k * (sum over the warps of path k), in a fixed order
            const float* col = slots + b * kSlotStride + rl;
            const float v = P.K == 2 ? path_sums<2, kWarps>(col, gk) : P.K == 3 ? path_sums<3, kWarps>(col, gk) : path_sums<1, kWarps>(col, gk);
            const float scaled = v * L.inv_unit;
            bad[i] = !(fabsf(scaled) < L.limit * (float)n_slices);       // inf or NaN: finite inputs cannot get here
            const long long q = bad[i] ? 0LL : __float2ll_rn(scaled);
            add[i] = (unsigned long long)(q + ((long long)n_slices << L.fix_bits)) + (1ULL << 55);
            const int row = rt * RABIT_TILE_ROWS + rl;
            if (arrivals == 1 && b < P.batch && row < L.M)               // a whole row tile: nobody else contributes
                L.y[(size_t)b * L.M + row] = bad[i] ? __ushort_as_half((unsigned short)0x7FFF) : __float2half_rn(v);
        }
        // all atomics of the thread back to back: nothing between them that could wait for an answer
#pragma unroll
        for (int i = 0; i < kPer; ++i) {
            const int o = tid + i * kGroupThreads, b = o >> 7, rl = o & 127;
            old[i] = 0ULL;
            if (b >= P.batch || arrivals == 1) continue;
            unsigned long long* word = L.acc + (size_t)b * L.Mp + rt * RABIT_TILE_ROWS + rl;
            if (!RABIT_IN_RANGE(rt * RABIT_TILE_ROWS + rl < L.Mp && b < RABIT_LUT_MAX_BATCH)) continue;
            if (bad[i]) atomicOr(word, 1ULL << 63);                      // sticky: the add below never carries into bit 63
            old[i] = atomicAdd(word, add[i]);
        }
#pragma unroll
        for (int i = 0; i < kPer; ++i) {
            const int o = tid + i * kGroupThreads, b = o >> 7, rl = o & 127;
            if (b >= P.batch || arrivals == 1) continue;
            if ((int)((old[i] >> 55) & 0xFFu) != arrivals - 1) continue;  // other segments of the row tile are still to come
            const unsigned long long sum = (old[i] & kSumMask) + (add[i] & kSumMask);
            const long long total = (long long)sum - ((long long)L.n_cs << L.fix_bits);
            const bool poisoned = bad[i] || (old[i] >> 63) != 0;
            const float v = poisoned ? __int_as_float(0x7FC00000) : __ll2float_rn(total) * L.unit;
            const int row = rt * RABIT_TILE_ROWS + rl;
            if (row < L.M) L.y[(size_t)b * L.M + row] = __float2half_rn(v);
            L.acc[(size_t)b * L.Mp + row] = 0ULL;                         // resting state for the next call
        }
        group_sync<kGroupThreads>(group);                              // the slots are free for the next segment
    }
    if (!waited) asm volatile("griddepcontrol.wait;" ::: "memory");
}

template <int GROUPS>
cudaError_t launch(const F16Params& P, int grid, int device, cudaStream_t stream) {
    static bool attr_done[64] = {false};
    const size_t smem = (size_t)(kThreads / 32) * (kRows * kSlotStride * sizeof(float) + kRing * 512);
    const int slot = device >= 0 && device < 64 ? device : 0;
    if (!attr_done[slot] || slot != device) {
        cudaError_t e = cudaFuncSetAttribute(rabit_gemv_f16_kernel<GROUPS>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        attr_done[slot] = true;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned int)grid);
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, rabit_gemv_f16_kernel<GROUPS>, P);
}

// Cuts the launch's (row tile, slice) pairs, in that order, into one contiguous range per SM, worked through by one group of
// 16 warps or cut once more into parts for two groups of 8.  A range costs its pairs and, in every group, kSegmentUs for each
// segment after its first (the last segment end is the same for everybody).  Two groups are cut where that is cheapest: in
// the middle, or at a row-tile boundary, so that neither group has more than one segment.  Ranges are grown greedily under a
// cost limit and the smallest limit that needs no more ranges than SMs is found by bisection, so that SMs whose range
// crosses boundaries get fewer pairs.  Two groups hide each other's segment ends (28672 x 8192 at 8 rows 42 -> 38 us, 11008 x 4096
// 13.4 -> 12.3) but publish more parts of row tiles and add up more partial sums where a range is short (4096 x 4096 6.6
// against 7.5): the cheaper estimate wins.  Remembered per thread by shape (a decoder calls the same few groups over and over).
struct Ranges {
    int n, K, batch, sms, shape[kMaxGroup][2];
    int groups, grid;
    F16Range range[kMaxRanges + 1];
};
struct Planner {
    int n, K, batch, groups;
    const int (*shape)[2];                               // [layer]: row tiles, slices
    long long pair0[kMaxGroup + 1], tile0[kMaxGroup + 1];
    double pair_us;

    Planner(int n, const int (*shape)[2], int K, int batch, int groups) : n(n), K(K), batch(batch), groups(groups), shape(shape), pair_us(8.0 * K * kTileClocks / 1900.0 * (K == 3 && groups == 2 ? kUneven3 : 1.0)) {
        pair0[0] = tile0[0] = 0;
        for (int l = 0; l < n; ++l) {
            pair0[l + 1] = pair0[l] + (long long)shape[l][0] * shape[l][1];
            tile0[l + 1] = tile0[l] + shape[l][0];
        }
    }
    // row tile of a pair, and its first pair and the first after it
    long long tile(long long u, long long* from = nullptr, long long* to = nullptr) const {
        int l = 0;
        while (l + 1 < n && u >= pair0[l + 1]) ++l;
        const long long t = (u - pair0[l]) / shape[l][1];
        if (from) *from = pair0[l] + t * shape[l][1];
        if (to) *to = pair0[l] + (t + 1) * shape[l][1];
        return tile0[l] + t;
    }
    double cost(long long a, long long b, long long* cut) const {        // of [a, b); two groups: the second starts at *cut
        *cut = b;
        const double whole = (double)(b - a) * pair_us;
        if (groups == 1 || b - a < 2) return whole * (groups == 1 ? 1.0 : kAlone) + kSegmentUs1 * (double)(tile(b - 1) - tile(a));
        double best = 1e300;
        auto consider = [&](long long m) {
            if (m <= a || m >= b) return;
            const double longer = (double)std::max(m - a, b - m), shorter = (double)std::min(m - a, b - m);
            const long long crossed = std::max(tile(m - 1) - tile(a), tile(b - 1) - tile(m));
            const double c = (2.0 * shorter + kAlone * (longer - shorter)) * pair_us + kSegmentUs2 * (double)crossed;
            if (c < best) { best = c; *cut = m; }
        };
        const long long mid = (a + b) / 2;
        long long from, to;
        tile(mid, &from, &to);
        consider(mid);
        consider(from);
        consider(to);
        return best;
    }
    // greedy ranges under the limit into out (starts, `groups` entries a range); their number, more than max_grid if that is exceeded
    int ranges(double limit, int max_grid, int* out) const {
        int grid = 0;
        long long cut;
        for (long long a = 0; a < pair0[n];) {
            if (grid == max_grid) return max_grid + 1;
            long long lo = a + 1, hi = std::min(pair0[n], a + (long long)(limit / pair_us) + 2);   // the longest range with cost <= limit
            while (lo < hi) {
                const long long mid = (lo + hi + 1) / 2;
                if (cost(a, mid, &cut) <= limit) lo = mid; else hi = mid - 1;
            }
            if (out) {
                cost(a, lo, &cut);
                out[groups * grid] = (int)a;
                if (groups == 2) out[2 * grid + 1] = (int)cut;
            }
            ++grid;
            a = lo;
        }
        return grid;
    }
    // the whole plan; returns its estimate
    double plan(int sms, Ranges* r) const {
        const int max_grid = (int)std::min<long long>(std::min(sms, kMaxRanges / groups), pair0[n]);
        double lo = 0.0, hi = (double)pair0[n] * pair_us * 2.0 + kSegmentUs1 * (double)tile0[n];
        for (int it = 0; it < 24; ++it) {
            const double mid = 0.5 * (lo + hi);
            if (ranges(mid, max_grid, nullptr) <= max_grid) hi = mid; else lo = mid;
        }
        int start[kMaxRanges + 1];
        r->groups = groups;
        r->grid = ranges(hi, max_grid, start);
        const int total = groups * r->grid;
        start[total] = (int)pair0[n];
        for (int q = 0; q <= kMaxRanges; ++q) r->range[q] = F16Range{q < total ? start[q] : (int)pair0[n], 0, 0, 0};
        long long parts = 0;                                             // segments that are not whole row tiles: these are published
        for (int q = 0; q < total; ++q) {
            if (start[q] == start[q + 1]) continue;
            auto touching = [&](long long u) {                           // non-empty ranges that touch the row tile of pair u, which this one does
                long long from, to;
                tile(u, &from, &to);
                int c = 1;
                for (int w = q; start[w] > from; --w) c += start[w - 1] < start[w];
                for (int w = q + 1; start[w] < to; ++w) c += start[w] < start[w + 1];
                return c;
            };
            const int first = touching(start[q]), last = touching(start[q + 1] - 1);
            r->range[q].first = (unsigned char)first;
            r->range[q].last = (unsigned char)last;
            parts += (first > 1) + (last > 1 && tile(start[q]) != tile(start[q + 1] - 1));
        }
        return hi + (parts ? kPublishUs + (double)parts * 128.0 * batch / 80.0 / 1900.0 : 0.0);
    }
};
const Ranges& plan_group(int n, const int (*shape)[2], int K, int batch, int sms) {
    static thread_local std::vector<Ranges> plans;
    for (const Ranges& pl : plans)
        if (pl.n == n && pl.K == K && pl.batch == batch && pl.sms == sms && std::memcmp(pl.shape, shape, sizeof(int) * 2 * n) == 0) return pl;
    Ranges one, two;
    std::memset(&one, 0, sizeof(one));
    one.n = n; one.K = K; one.batch = batch; one.sms = sms;
    std::memcpy(one.shape, shape, sizeof(int) * 2 * n);
    two = one;
    const double us1 = Planner(n, shape, K, batch, 1).plan(sms, &one), us2 = Planner(n, shape, K, batch, 2).plan(sms, &two);
    if (plans.size() >= 256) plans.clear();
    plans.push_back(us2 < us1 ? two : one);
    return plans.back();
}

}  // namespace

// Host-only view of the work split (for tests): two entries per CTA, the starts of its two groups' ranges (with one group the
// second is empty), for a K-path layer of M x N at `batch` rows on `sms` SMs; bound_out receives 2 * grid + 1 values, the last being
// the number of pairs.
int rabit_gemv_f16_plan(int K, int M, int N, int batch, int sms, int* bound_out, int max_out) {
    if (K < 1 || K > RABIT_MAX_K || M < 1 || N < 32 || (N % 32) != 0 || batch < 1 || batch > RABIT_MAX_GEMV_BATCH || sms < 1) return -1;
    const long long n_rt = ((long long)M + RABIT_TILE_ROWS - 1) / RABIT_TILE_ROWS, n_cs = ((long long)N + RABIT_LUT_COLS - 1) / RABIT_LUT_COLS;
    if (n_cs > RABIT_LUT_MAX_SLICES || n_rt * n_cs >= kMaxPairs) return -1;
    const int shape[1][2] = {{(int)n_rt, (int)n_cs}};
    const Ranges& pl = plan_group(1, shape, K, batch, sms);
    if (max_out < 2 * pl.grid + 1) return -1;
    for (int c = 0; c < pl.grid; ++c) {
        bound_out[2 * c] = pl.range[pl.groups * c].start;
        bound_out[2 * c + 1] = pl.range[pl.groups * c + 1].start;
    }
    bound_out[2 * pl.grid] = (int)(n_rt * n_cs);
    return pl.grid;
}

bool rabit_gemv_f16_supports(const rabit_layer& L, int batch) {
    if (batch < 1 || batch > kRows) return false;
    if (L.geom.n_cs > RABIT_LUT_MAX_SLICES || L.d_acc == nullptr) return false;
    if ((long long)L.geom.n_rt * L.geom.K * L.geom.n_ct * 32 >= (1LL << 31)) return false;   // 32-bit tile offsets in the kernel
    return (long long)L.geom.n_rt * L.geom.n_cs < kMaxPairs;
}

bool rabit_gemv_f16_group_supports(const rabit_layer* const* layers, int n_layers, int batch) {
    if (n_layers < 1 || n_layers > kMaxGroup) return false;
    long long pairs = 0;
    for (int l = 0; l < n_layers; ++l) {
        pairs += (long long)layers[l]->geom.n_rt * layers[l]->geom.n_cs;
        if (pairs >= kMaxPairs || !rabit_gemv_f16_supports(*layers[l], batch) || layers[l]->geom.K != layers[0]->geom.K) return false;
        for (int m = 0; m < l; ++m)
            if (layers[m] == layers[l]) return false;                    // one layer twice would share its accumulate words
    }
    return true;
}

// One launch for n_layers independent layers of equal K, 1..8 batch rows (x_l: [batch][N_l], y_l: [batch][M_l]).
cudaError_t rabit_launch_gemv_f16_group(const rabit_layer* const* layers, int n_layers, const void* const* xs, void* const* ys, int batch, cudaStream_t stream) {
    if (!rabit_gemv_f16_group_supports(layers, n_layers, batch)) return cudaErrorInvalidValue;
    const int K = layers[0]->geom.K, sms = layers[0]->sm_count > 0 ? layers[0]->sm_count : 148;
    int shape[kMaxGroup][2];
    for (int l = 0; l < n_layers; ++l) { shape[l][0] = layers[l]->geom.n_rt; shape[l][1] = layers[l]->geom.n_cs; }
    const Ranges& pl = plan_group(n_layers, shape, K, batch, sms);
    F16Params P;
    P.n_layers = n_layers;
    P.K = K;
    P.batch = batch;
    P.four = 4u;
    P.two_pow_8 = 256u;
    int pairs = 0;
    for (int l = 0; l < kMaxGroup; ++l) {
        P.pair0[l] = pairs;
        if (l >= n_layers) { P.layer[l] = P.layer[0]; continue; }
        const rabit_layer& Ly = *layers[l];
        const RabitGeom& G = Ly.geom;
        F16Layer& D = P.layer[l];
        D.tiles = Ly.d_bits;
        D.g = (const __half*)Ly.d_g;
        D.h = (const __half*)Ly.d_h;
        D.x = (const __half*)xs[l];
        D.y = (__half*)ys[l];
        D.acc = Ly.d_acc;
        D.status = Ly.d_status;
        D.M = G.M; D.N = G.N; D.Mp = G.Mp; D.n_rt = G.n_rt; D.n_ct = G.n_ct; D.n_cs = G.n_cs;
        D.fix_bits = G.fix_bits;
        D.unit = ldexpf(1.f, G.unit_exp);
        D.inv_unit = ldexpf(1.f, -G.unit_exp);
        D.limit = ldexpf(1.f, G.fix_bits);
        pairs += G.n_rt * G.n_cs;
    }
    std::memcpy(P.range, pl.range, sizeof(P.range));
    return pl.groups == 1 ? launch<1>(P, pl.grid, layers[0]->device, stream) : launch<2>(P, pl.grid, layers[0]->device, stream);
}

cudaError_t rabit_launch_gemv_f16(const rabit_layer& L, const void* x, void* y, int batch, cudaStream_t stream) {
    const rabit_layer* one = &L;
    return rabit_launch_gemv_f16_group(&one, 1, &x, &y, batch, stream);
}
