// Decode GEMV for 3..16 batch rows: the batch sits in the N dimension of an f16 tensor-core MMA.
//
//   y[b][i] = sum_k g_k[i] * sum_j (B_k[i][j] h_k[j]) * x[b][j]                              (Section 4.1, Eq. 2)
//
// The table-driven kernel (rabit_gemv_lut.cu) pays per batch row; the integer tensor-core GEMV spends four of an MMA's
// eight columns per batch row and needs a pass over x first.  Here the A operand of mma.sync.m16n8k16 is +-h_k expanded in
// registers from the sign tiles (the weight bit flips the sign bit of the fp16 input scale: exact), B is x as it is, the
// accumulators are fp32: products are exact, 8 batch rows per MMA and 16 with a second MMA on the same A, no digits, no
// scale search.  The cost is that of the expansion and does not depend on the batch.
//
// Expansion.  Shifts, byte permutes and logic instructions all issue on the half-rate integer pipe of an SM sub-partition
// (16 lanes per clock), and that pipe, not the tensor pipe, bounds this kernel.  So an A register (two fp16 values) costs
// ONE logic instruction there, (v & 0x80008000) ^ h, and the shift that brings the two weight bits to bits 15 and 31 is a
// multiplication by a power of two on the multiply-add pipe: v = w * 2^s, where the factor comes from a kernel parameter
// so that the compiler keeps it a multiplication.  The two bits must be 16 apart in the word, i.e. two columns apart:
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
// Work split.  The layer is n_rt row tiles x n_cs slices of 256 columns.  Every row tile is cut into m equal units and a CTA
// (16 warps, one CTA per SM) takes j consecutive units (split_layer on the host chooses m and j by a cost model).  The part
// of a CTA's range inside one row tile is a segment.  Warp w works on path w % K and shares the column tiles of the segment
// with the other warps of that path.  A warp streams its tiles through a ring of its own in shared memory with asynchronous
// 16-byte copies (one per lane and tile, each lane reads back only what it copied itself, so no barrier is involved),
// kRing - 1 tiles ahead: with 16 warps per SM that keeps about 56 KB per SM in flight, which is what the HBM latency needs
// (with the tiles prefetched into registers, two to four per warp, the kernel ran at the speed of its memory latency, 1.1
// to 1.7 TB/s).  At the end of a segment every warp writes its accumulators to its own slot of shared memory and the CTA adds
// the slots path by path in a fixed order (deterministic), applying g_k to each path's sum.  A segment that is a whole row
// tile stores y.  Otherwise every output goes, as in the table-driven kernel, into the row's 64-bit accumulate word with one
// integer atomic (fixed-point grid of the packer, arrival count in bits 55..62, bit 63 = non-finite); the thread whose add
// completes a row (the count reaches the number of segments of that row tile) rounds it to fp16, stores y and clears the
// word.  A contribution that covers s slices is shifted by s * 2^fix_bits, so the total shift is the same n_cs * 2^fix_bits
// for every split.  Nothing waits for another CTA.
//
// What bounds it (B200, clocks per 512-byte tile and SM): 75 at up to eight batch rows and 105 at sixteen in the steady state,
// of which the loads of x and h are 10 %; the rest is 16 or 32 MMAs of about 2 clocks and 128 half-rate integer operations,
// which hardly overlap.  Segment ends are what a split can save: an arrival count found by searching a table of range
// bounds in constant memory, cold in every launch, cost 1 us at each, publishing 16 rows from every SM 2 to 3 us.
#include <cuda_fp16.h>

#include <algorithm>
#include <cstring>
#include <vector>

#include "rabit_internal.h"

namespace {

constexpr int kWarps = 16;
constexpr int kThreads = kWarps * 32;
constexpr int kRing = 8;                               // sign tiles a warp keeps in flight or in use (a power of two)
constexpr long long kMaxPairs = 1LL << 30;
constexpr int kMaxGroup = 8;
constexpr int kSlotStride = 128 + 4;                  // floats per batch row of a slot: the pad spreads a warp's store over all banks
constexpr unsigned long long kSumMask = (1ULL << 55) - 1;

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
    int cta0;                       // the layer's first CTA
    int m, j;                       // units per row tile, units per CTA
    int pad_;
};
static_assert(sizeof(F16Layer) % 4 == 0 && sizeof(F16Layer) <= 128, "F16Layer is copied to shared memory by one warp, a word per lane");
struct F16Params {
    int n_layers, K, batch;
    uint32_t two, two_pow_8;        // 2 and 256: multipliers the compiler cannot fold into shifts
    F16Layer layer[kMaxGroup];
};

// First pair of a unit: unit q of row tile t starts at slice q n_cs / m of it.  (Host and device.)
__host__ __device__ __forceinline__ int unit_start(int unit, int m, int n_cs) {
    const int t = unit / m;
    return t * n_cs + (int)((long long)(unit - t * m) * n_cs / m);
}

// Checked build (-DRABIT_CHECKED, python paper_2602_05367_b200/build.py --checked): every index that addresses global or
// shared memory is compared with its range first; a violation is recorded in the layer's status word and the access is
// skipped (nothing traps).  In the ordinary build the checks compile to nothing.
#ifdef RABIT_CHECKED
#define RABIT_IN_RANGE(cond) ((cond) ? true : (atomicExch(L.status, 2u), false))
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
template <int KK, int NH>
__device__ __forceinline__ float path_sums(const float* col, const __half (&g)[RABIT_MAX_K]) {
    float sk[KK];
#pragma unroll
    for (int kk = 0; kk < KK; ++kk) sk[kk] = 0.f;
#pragma unroll
    for (int wv = 0; wv < kWarps; ++wv) sk[wv % KK] += col[(size_t)wv * (NH * 8 * kSlotStride)];
    float v = 0.f;
#pragma unroll
    for (int kk = 0; kk < KK; ++kk) v = fmaf(__half2float(g[kk]), sk[kk], v);
    return v;
}

// NH = halves of the batch (8 rows each) a pass carries.
template <int NH>
__global__ void __launch_bounds__(kThreads, 1)
rabit_gemv_f16_kernel(const __grid_constant__ F16Params P) {
    extern __shared__ __align__(16) float smem_f[];                      // [kWarps][NH * 8][kSlotStride] partial outputs, then the warps' rings
    [[maybe_unused]] constexpr int kFloats = kWarps * NH * 8 * kSlotStride + kWarps * kRing * 128;
    __shared__ F16Layer layer_copy;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int gq = lane >> 2, tq = lane & 3;
    float* slots = smem_f;
    // the lane's 16 bytes of ring slot 0 of its warp; slot r is r * 512 bytes further
    const uint32_t ring = (uint32_t)__cvta_generic_to_shared(slots) + (uint32_t)(kWarps * NH * 8 * kSlotStride * sizeof(float)) +
                          (uint32_t)((warp * kRing * 32 + lane) * 16);

    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    bool waited = false;
    // the launch parameters sit in constant memory, cold in every launch: copied once, before the dependency wait
    if (warp == 0) {
        int li = 0;
        while (li + 1 < P.n_layers && (int)blockIdx.x >= P.layer[li + 1].cta0) ++li;
        if (lane < (int)(sizeof(F16Layer) / 4)) reinterpret_cast<uint32_t*>(&layer_copy)[lane] = reinterpret_cast<const uint32_t*>(&P.layer[li])[lane];
    }
    __syncthreads();
    const F16Layer& L = layer_copy;
    const __half *const h_base = L.h, *const x_base = L.x;               // (what the loop needs of the layer, in registers)
    const int n_ct = L.n_ct, n_cs = L.n_cs;

    // every warp works on ONE path: path k = warp % K, and the column tiles of a segment are dealt out among the
    // warps of that path (K = 3: six, five and five warps)
    const int k = warp % P.K;
    const int n_same = (kWarps - k + P.K - 1) / P.K, j0 = warp / P.K;
    const int hk = k * L.N + 4 * tq;                                      // element offsets (K * N and 16 * N fit 31 bits: N <= 65280)
    int xb[NH];
#pragma unroll
    for (int hf = 0; hf < NH; ++hf)                                      // lanes beyond the batch read its last row; their columns are never stored
        xb[hf] = min(8 * hf + gq, P.batch - 1) * L.N + 4 * tq;

    // A segment: row tile rt, column tiles [ct0, c1) of which this warp takes every n_same-th, starting at ct0.
    struct Segment {
        int rt, n_slices, c1, ct0, n_my;
        const uint4* wsrc;                                               // the warp's first tile (this lane's 16 bytes)
    };
    const int c_rel = (int)blockIdx.x - L.cta0, n_units = L.n_rt * L.m;
    int u = unit_start(c_rel * L.j, L.m, n_cs);
    const int u_end = unit_start(min(n_units, (c_rel + 1) * L.j), L.m, n_cs);
    auto next_segment = [&]() {                                          // the segment that starts at pair u; advances u
        Segment sg;
        sg.rt = u / n_cs;
        const int s0 = u - sg.rt * n_cs;
        const int s1 = min(n_cs, s0 + (u_end - u));
        u += s1 - s0;
        sg.n_slices = s1 - s0;
        sg.c1 = min(n_ct, s1 * 8);                                     // a slice is eight column tiles
        sg.ct0 = s0 * 8 + j0;
        sg.n_my = sg.ct0 < sg.c1 ? (sg.c1 - sg.ct0 + n_same - 1) / n_same : 0;
        sg.wsrc = L.tiles + (size_t)(sg.rt * P.K + k) * n_ct * 32 + sg.ct0 * 32 + lane;
        return sg;
    };
    auto prefill = [&](const Segment& sg) {                              // the first kRing - 1 tiles of the warp; weights never depend on the stream's past
#pragma unroll
        for (int i = 0; i < kRing - 1; ++i)
            copy_async_16(ring + i * 512, sg.wsrc + (size_t)i * n_same * 32,
                          i < sg.n_my && RABIT_IN_RANGE(sg.wsrc + (size_t)i * n_same * 32 >= L.tiles &&
                                                        sg.wsrc + (size_t)i * n_same * 32 < L.tiles + (size_t)L.n_rt * P.K * n_ct * 32));
    };
    bool more = u < u_end;
    Segment sg;
    if (more) {
        sg = next_segment();
        prefill(sg);
    }
    while (more) {
        const int rt = sg.rt, ct0 = sg.ct0, n_my = sg.n_my;
        const uint4* wsrc = sg.wsrc;
        float acc[8][NH][4];
#pragma unroll
        for (int p = 0; p < 8; ++p)
#pragma unroll
            for (int hf = 0; hf < NH; ++hf)
#pragma unroll
                for (int e = 0; e < 4; ++e) acc[p][hf][e] = 0.f;

        // input scales and activations of the lane's four columns of k-step kh of column tile ct, as loaded (columns 0,1 | 2,3)
        auto fetch_hx = [&](int ct, int kh, uint2& fh, uint2 (&fx)[NH]) {
            const int off = ct * 32 + 16 * kh;
            if (!RABIT_IN_RANGE(off >= 0 && hk + off + 4 <= P.K * L.N)) return;
            fh = __ldg(reinterpret_cast<const uint2*>(h_base + hk + off));
#pragma unroll
            for (int hf = 0; hf < NH; ++hf)
                if (RABIT_IN_RANGE(xb[hf] + off + 4 <= P.batch * L.N)) fx[hf] = __ldcg(reinterpret_cast<const uint2*>(x_base + xb[hf] + off));
        };

        __half gk[RABIT_MAX_K];                                           // output scales of the thread's row (the same row for all its outputs), loaded long before they are used
#pragma unroll
        for (int kk = 0; kk < RABIT_MAX_K; ++kk)
            gk[kk] = kk < P.K ? L.g[(size_t)kk * L.Mp + rt * RABIT_TILE_ROWS + (tid & 127)] : __half();
        // weights kRing - 1 tiles ahead (HBM latency), scales and activations one tile ahead, k-step by k-step in place
        if (!waited) {
            asm volatile("griddepcontrol.wait;" ::: "memory");            // x, y and the accumulate words only after this
            waited = true;
        }
        uint2 fh[2], fx[2][NH];
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
                    uint32_t b0[NH], b1[NH];
#pragma unroll
                    for (int hf = 0; hf < NH; ++hf) {
                        b0[hf] = prmt(fx[kh][hf].x, fx[kh][hf].y, 0x5410);
                        b1[hf] = prmt(fx[kh][hf].x, fx[kh][hf].y, 0x7632);
                    }
                    fetch_hx(ct_next, kh, fh[kh], fx[kh]);                // the same k-step of the warp's next tile, in place
                    // u = w * 2^(7-p): bit p of bytes 1 and 3 -> bits 15 and 31;  v = u * 2^8: the same for bytes 0 and 2
                    uint32_t ul = w[2 * kh], uh = w[2 * kh + 1];
                    uint32_t vl = mul_lo(ul, P.two_pow_8), vh = mul_lo(uh, P.two_pow_8);
#pragma unroll
                    for (int p = 7; p >= 0; --p) {
                        const uint32_t a0 = flip(vl, h02), a1 = flip(vh, h02), a2 = flip(ul, h13), a3 = flip(uh, h13);
#pragma unroll
                        for (int hf = 0; hf < NH; ++hf) mma_f16(acc[p][hf], a0, a1, a2, a3, b0[hf], b1[hf]);
                        if (p > 0) {
                            ul = mul_lo(ul, P.two); uh = mul_lo(uh, P.two);
                            vl = mul_lo(vl, P.two); vh = mul_lo(vh, P.two);
                        }
                    }
                }
            }
        }
        copy_async_wait<0>();
        // the next segment's first tiles set off now: they cross HBM while this segment is added up
        const int n_slices = sg.n_slices;
        more = u < u_end;
        if (more) {
            sg = next_segment();
            prefill(sg);
        }
        constexpr int kPer = NH * 8 * 128 / kThreads;                         // outputs per thread (2 or 4)
        // ---- the warp's partial outputs -> its slot; slot layout [batch row][row of the tile]
        float* mine = slots + (size_t)warp * (NH * 8 * kSlotStride);
        const bool slot_ok = RABIT_IN_RANGE(mine + (NH * 8 - 1) * kSlotStride + 127 < smem_f + kFloats);
#pragma unroll
        for (int p = 0; p < 8; ++p)
#pragma unroll
            for (int hf = 0; hf < NH; ++hf) {
                if (!slot_ok) break;
                const int b = 8 * hf + 2 * tq, row = 16 * p + gq;
                mine[(b) * kSlotStride + row] = acc[p][hf][0];
                mine[(b + 1) * kSlotStride + row] = acc[p][hf][1];
                mine[(b) * kSlotStride + row + 8] = acc[p][hf][2];
                mine[(b + 1) * kSlotStride + row + 8] = acc[p][hf][3];
            }
        __syncthreads();
        // ---- fixed-order sum over the warps, then one atomic per output of the segment
        const int arrivals = (rt * L.m + L.m - 1) / L.j - rt * L.m / L.j + 1;    // segments of this row tile: the CTAs whose units touch it
        // (thread t owns row t & 127 of the tile and the batch rows (t >> 7) + 4 i; rows beyond the batch are computed from
        // whatever their MMA columns held and dropped)
        unsigned long long old[kPer], add[kPer];
        bool bad[kPer];
#pragma unroll
        for (int i = 0; i < kPer; ++i) {
            const int o = tid + i * kThreads, b = o >> 7, rl = o & 127;
            // sum_k g_k * (sum over the warps of path k), in a fixed order
            const float* col = slots + b * kSlotStride + rl;
            const float v = P.K == 2 ? path_sums<2, NH>(col, gk) : P.K == 3 ? path_sums<3, NH>(col, gk) : path_sums<1, NH>(col, gk);
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
            const int o = tid + i * kThreads, b = o >> 7, rl = o & 127;
            old[i] = 0ULL;
            if (b >= P.batch || arrivals == 1) continue;
            unsigned long long* word = L.acc + (size_t)b * L.Mp + rt * RABIT_TILE_ROWS + rl;
            if (!RABIT_IN_RANGE(rt * RABIT_TILE_ROWS + rl < L.Mp && b < RABIT_LUT_MAX_BATCH)) continue;
            if (bad[i]) atomicOr(word, 1ULL << 63);                      // sticky: the add below never carries into bit 63
            old[i] = atomicAdd(word, add[i]);
        }
#pragma unroll
        for (int i = 0; i < kPer; ++i) {
            const int o = tid + i * kThreads, b = o >> 7, rl = o & 127;
            if (b >= P.batch || arrivals == 1) continue;
            if ((int)((old[i] >> 55) & 0xFFu) != arrivals - 1) continue;  // other segments of the row tile are still to come
            const unsigned long long sum = (old[i] & kSumMask) + (add[i] & kSumMask);
            const long long total = (long long)sum - ((long long)n_cs << L.fix_bits);
            const bool poisoned = bad[i] || (old[i] >> 63) != 0;
            const float v = poisoned ? __int_as_float(0x7FC00000) : __ll2float_rn(total) * L.unit;
            const int row = rt * RABIT_TILE_ROWS + rl;
            if (row < L.M) L.y[(size_t)b * L.M + row] = __float2half_rn(v);
            L.acc[(size_t)b * L.Mp + row] = 0ULL;                         // resting state for the next call
        }
        __syncthreads();                                               // the slots are free for the next segment
    }
    if (!waited) asm volatile("griddepcontrol.wait;" ::: "memory");
}

template <int NH>
cudaError_t launch(const F16Params& P, int grid, int device, cudaStream_t stream) {
    static bool attr_done[64] = {false};
    const size_t smem = (size_t)kWarps * NH * 8 * kSlotStride * sizeof(float) + (size_t)kWarps * kRing * 512;
    const int slot = device >= 0 && device < 64 ? device : 0;
    if (!attr_done[slot] || slot != device) {
        cudaError_t e = cudaFuncSetAttribute(rabit_gemv_f16_kernel<NH>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        attr_done[slot] = true;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, rabit_gemv_f16_kernel<NH>, P);
}

struct Split {
    int m, j, n_cta;
    double us;                                                           // estimate
};

// Cuts the n_rt * n_cs (row tile, slice) pairs into at most `ctas` ranges: every row tile into m equal units, j consecutive units
// per CTA, for the m with the smallest estimate.  m = 1 is whole row tiles (no atomics), m = ctas / n_rt equal parts of
// one, larger m ranges that cross row tiles.  The estimate, from timelines on B200: a tile takes 78 (up to eight batch rows)
// or 108 clocks, a segment end inside a range 1.5 us, publishing parts of row tiles 0.6 us plus 128 * batch words per part
// at 80 words per clock over the whole GPU.
Split split_layer(int n_rt, int n_cs, int K, int batch, int ctas) {
    const double pair_us = 8.0 * K * (batch > 8 ? 108.0 : 78.0) / 1900.0;
    Split best = {1, 1, 0, 1e300};
    for (int m = 1; m <= n_cs; ++m) {
        const long long units = (long long)n_rt * m;
        const int j = (int)((units + ctas - 1) / ctas), n = (int)((units + j - 1) / j);
        // ranges repeat after lcm(m, j) units, so the first few CTAs show the worst one
        double worst = 0.0;
        long long parts = 0;                                             // segments that are not whole row tiles
        const int look = std::min(n, m + 1);
        for (int c = 0; c < look; ++c) {
            const long long a = unit_start(c * j, m, n_cs), b = unit_start((int)std::min<long long>(units, (long long)(c + 1) * j), m, n_cs);
            const long long segments = (b - 1) / n_cs - a / n_cs + 1;
            const int cut = (a % n_cs != 0) + (b % n_cs != 0);
            parts += segments == 1 && cut == 2 ? 1 : cut;
            worst = std::max(worst, (double)(b - a) * pair_us + 1.5 * (double)(segments - 1));
        }
        const double us = worst + (parts ? 0.6 + (double)parts * n / look * 128.0 * batch / 80.0 / 1900.0 : 0.0);
        if (us < best.us) best = Split{m, j, n, us};
        if (units >= 64LL * ctas) break;                                 // finer cuts change nothing any more
    }
    return best;
}

// A launch's split.  CTAs in proportion to the pairs, at least one per layer; then one at a time from what is left, or from
// the layer that would finish first, to the one that would finish last while that helps.  Remembered per thread by shape
// (a decoder calls the same few groups over and over).
struct GroupPlan {
    int n, K, batch, sms, shape[kMaxGroup][2];
    Split split[kMaxGroup];
};
GroupPlan plan_group(int n, const int (*shape)[2], int K, int batch, int sms) {
    static thread_local std::vector<GroupPlan> plans;
    for (const GroupPlan& pl : plans)
        if (pl.n == n && pl.K == K && pl.batch == batch && pl.sms == sms && std::memcmp(pl.shape, shape, sizeof(int) * 2 * n) == 0) return pl;
    GroupPlan pl;
    std::memset(&pl, 0, sizeof(pl));
    pl.n = n; pl.K = K; pl.batch = batch; pl.sms = sms;
    std::memcpy(pl.shape, shape, sizeof(int) * 2 * n);
    const int ctas = std::max(sms, n);
    long long total = 0;
    for (int l = 0; l < n; ++l) total += (long long)shape[l][0] * shape[l][1];
    int give[kMaxGroup], given = 0;
    for (int l = 0; l < n; ++l) {
        give[l] = (int)std::max<long long>(1, (long long)ctas * shape[l][0] * shape[l][1] / total);
        given += give[l];
    }
    while (given > ctas) {                                               // (many tiny layers beside a large one)
        int big = 0;
        for (int l = 1; l < n; ++l) if (give[l] > give[big]) big = l;
        --give[big]; --given;
    }
    auto cut = [&](int l, int c) { return split_layer(shape[l][0], shape[l][1], K, batch, c); };
    for (int l = 0; l < n; ++l) pl.split[l] = cut(l, n == 1 ? ctas : give[l]);
    for (int iter = 0; iter < 24 && n > 1; ++iter) {
        int hi = 0, lo = -1;
        for (int l = 1; l < n; ++l) if (pl.split[l].us > pl.split[hi].us) hi = l;
        bool better = false;
        for (int take = 1; take <= ctas - given && !better; ++take) {    // the smallest number of spare CTAs that helps the slowest layer
            const Split up = cut(hi, give[hi] + take);
            if (up.us < pl.split[hi].us - 1e-9) { give[hi] += take; given += take; pl.split[hi] = up; better = true; }
        }
        for (int l = 0; l < n && !better; ++l)
            if (l != hi && give[l] > 1 && (lo < 0 || pl.split[l].us < pl.split[lo].us)) lo = l;
        if (!better && lo >= 0) {
            const Split up = cut(hi, give[hi] + 1), down = cut(lo, give[lo] - 1);
            if (std::max(up.us, down.us) < pl.split[hi].us - 1e-9) {
                give[hi] += 1; give[lo] -= 1;
                pl.split[hi] = up; pl.split[lo] = down;
                better = true;
            }
        }
        if (!better) break;
    }
    if (plans.size() >= 256) plans.clear();
    plans.push_back(pl);
    return pl;
}

}  // namespace

// Host-only view of the work split (for tests): two entries per CTA, the start of its range and its end (a range is not divided
// any further: the second part is empty), for a K-path layer of M x N at `batch` rows on `sms` SMs; bound_out receives
// 2 * grid + 1 values, the last being the number of pairs.
int rabit_gemv_f16_plan(int K, int M, int N, int batch, int sms, int* bound_out, int max_out) {
    if (K < 1 || K > RABIT_MAX_K || M < 1 || N < 32 || (N % 32) != 0 || batch < 1 || batch > RABIT_MAX_GEMV_BATCH || sms < 1) return -1;
    const long long n_rt = ((long long)M + RABIT_TILE_ROWS - 1) / RABIT_TILE_ROWS, n_cs = ((long long)N + RABIT_LUT_COLS - 1) / RABIT_LUT_COLS;
    if (n_cs > RABIT_LUT_MAX_SLICES || n_rt * n_cs >= kMaxPairs) return -1;
    const int shape[1][2] = {{(int)n_rt, (int)n_cs}};
    const Split sp = plan_group(1, shape, K, batch, sms).split[0];
    if (max_out < 2 * sp.n_cta + 1) return -1;
    for (int c = 0; c < sp.n_cta; ++c) {
        bound_out[2 * c] = unit_start(c * sp.j, sp.m, (int)n_cs);
        bound_out[2 * c + 1] = unit_start((int)std::min(n_rt * sp.m, (long long)(c + 1) * sp.j), sp.m, (int)n_cs);
    }
    bound_out[2 * sp.n_cta] = (int)(n_rt * n_cs);
    return sp.n_cta;
}

bool rabit_gemv_f16_supports(const rabit_layer& L, int batch) {
    if (batch < 1 || batch > RABIT_MAX_GEMV_BATCH) return false;
    if (L.geom.n_cs > RABIT_LUT_MAX_SLICES || L.d_acc == nullptr) return false;
    if ((long long)L.geom.n_rt * L.geom.K * L.geom.n_ct * 32 >= (1LL << 31)) return false;   // 32-bit tile offsets in the kernel
    return (long long)L.geom.n_rt * L.geom.n_cs < kMaxPairs;
}

bool rabit_gemv_f16_group_supports(const rabit_layer* const* layers, int n_layers, int batch) {
    if (n_layers < 1 || n_layers > kMaxGroup) return false;
    for (int l = 0; l < n_layers; ++l) {
        if (!rabit_gemv_f16_supports(*layers[l], batch) || layers[l]->geom.K != layers[0]->geom.K) return false;
        for (int m = 0; m < l; ++m)
            if (layers[m] == layers[l]) return false;                    // one layer twice would share its accumulate words
    }
    return true;
}

// One launch for n_layers independent layers of equal K, 1..16 batch rows (x_l: [batch][N_l], y_l: [batch][M_l]).
cudaError_t rabit_launch_gemv_f16_group(const rabit_layer* const* layers, int n_layers, const void* const* xs, void* const* ys, int batch, cudaStream_t stream) {
    if (!rabit_gemv_f16_group_supports(layers, n_layers, batch)) return cudaErrorInvalidValue;
    const int K = layers[0]->geom.K, sms = layers[0]->sm_count > 0 ? layers[0]->sm_count : 148;
    int shape[kMaxGroup][2];
    for (int l = 0; l < n_layers; ++l) { shape[l][0] = layers[l]->geom.n_rt; shape[l][1] = layers[l]->geom.n_cs; }
    const GroupPlan pl = plan_group(n_layers, shape, K, batch, sms);
    F16Params P;
    P.n_layers = n_layers;
    P.K = K;
    P.batch = batch;
    P.two = 2u;
    P.two_pow_8 = 256u;
    int at = 0;
    for (int l = 0; l < n_layers; ++l) {
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
        D.cta0 = at; D.m = pl.split[l].m; D.j = pl.split[l].j;
        D.pad_ = 0;
        at += pl.split[l].n_cta;
    }
    for (int l = n_layers; l < kMaxGroup; ++l) P.layer[l] = P.layer[0];
    return batch <= 8 ? launch<1>(P, at, layers[0]->device, stream) : launch<2>(P, at, layers[0]->device, stream);
}

cudaError_t rabit_launch_gemv_f16(const rabit_layer& L, const void* x, void* y, int batch, cudaStream_t stream) {
    const rabit_layer* one = &L;
    return rabit_launch_gemv_f16_group(&one, 1, &x, &y, batch, stream);
}
