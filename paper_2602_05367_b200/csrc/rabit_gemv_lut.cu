// Decode GEMV by table look-up (batch 1..2 per launch): the HBM-bound form of the layer
//
//   y[b][i] = sum_k g_k[i] * sum_j B_k[i][j] * t_k[b][j],   t_k[b][j] = h_k[j] * x[b][j]     (Section 4.1, Eq. 2)
//
// At one bit per weight a sign-select add per weight costs more instruction issue slots than HBM
// leaves time for (about 180 weight bits arrive per clock per SM, 128 lane-instructions issue).  The
// signs of eight consecutive input columns of one row are one byte of the packed image (look-up blocks,
// rabit_layout.h), and that byte indexes a 256-entry table of the partial sums  sum_{b<8} (+-) t[8c+b]
// built once per CTA in shared memory: one byte permute (the address), one shared-memory load and one
// fp32 add per EIGHT weights.  The input scale h_k is applied once per table (t = h * x), the signed
// accumulation is the sum of table entries in fp32 registers, and every weight bit is read once.
// Measured on B200, clocks per 2 KB block and SM on a layer of 114688 x 8192: the look-ups alone 67 (64 conflict-free wavefronts of
// the shared-memory pipe; 8.9 TB/s over 148 SMs, above what HBM delivers), the whole loop 118 with one batch row (5.1 TB/s).
// One row: without the loads of the next blocks 99, without the atomics 115.5,
// without the look-ups 106: the loop waits for its weights, of which at most one block per warp (32 KB per SM) is under way.
// Two rows: a look-up reads both rows' sums (8 bytes, 128 wavefronts a block whichever way) and one add takes both: 12 instructions instead
// of 20 per word and path, and the next block's weights are loaded beside the look-ups instead of behind them.  28672 x 8192
// 22.8 -> 20.9 us, 22016 x 4096 10.65 -> 9.95, 12288 x 4096 7.55 -> 7.0, one path 22016 x 4096 9.2 -> 7.5.  (The 8-byte look-ups without the
// earlier loads: one path 8.2, two paths 28672 x 8192 24.1: warps then wait for weights.  The packed add for one row: two paths 3 % slower.)
// One row: 28672 x 8192 15.0 us.
//
// Work split.  The layer is a grid of blocks (32 rows x 256 columns x K paths, K KB each) stored
// slice-major; CTA c owns a contiguous range of block positions (cut on the host so that all CTAs cost
// the same: so much per block, so much per table), which is one contiguous byte range.  A range that
// crosses into the next 256-column slice rebuilds its table there.  One CTA per SM, 16 warps:
//   * before the dependency wait (weights do not depend on the previous kernel in the stream, so this
//     overlaps its tail under programmatic dependent launch): every warp loads its first block into
//     registers and the input scales of the first table are read (a bulk L2 prefetch of the CTA's whole
//     range at this point was measured and made the kernel 8-10 % slower: the loads then meet their own
//     prefetch in L2);
//   * after the wait: x of the slice is read, the table is built (lane = byte group, warp = path x upper
//     three index bits; 32 entries each by doubling), and the warps take the blocks round-robin, lane =
//     row.  A lane holds its 16*K weight words in registers (128-bit streaming loads; the next block's come into the
//     registers behind the look-ups, and none after a warp's last block: reloading it there, unused, cost a 7B decoder
//     layer 22.0 instead of 21.3 us; two blocks ahead 23.1, rings filled by bulk copies 22.8 to 24.5), walks the 32 byte groups of
//     its row in an order rotated by its lane index (so the 32 look-ups of a warp step hit 32 banks), and
//     ends with  p = sum_k g_k[row] * s_k;
//   * reduction over the slices of a row, without a second pass, a fence or a wait: p is rounded to a
//     fixed-point grid that the packer sized so that no finite fp16 input can overflow it, and added with
//     ONE 64-bit integer atomic to the row's accumulate word, which also counts arrivals (bits 55..62).
//     The lane whose add returns "all other slices were here" owns the complete sum (old value + its own
//     term): it rounds once to fp16, stores y and puts the word back to zero.  Integer addition commutes,
//     so results do not depend on arrival order; a non-finite partial sum sets bit 63 (NaN output).
// No thread ever waits for another CTA, and the only waits inside a CTA are barriers of its own warps.
#include <cuda_fp16.h>

#include <algorithm>
#include <cstring>
#include <type_traits>
#include <vector>

#include "rabit_internal.h"

namespace {

constexpr int kWarps = 16;
constexpr int kThreads = kWarps * 32;
constexpr int kMaxGrid = 160;
constexpr int kMaxGroup = 8;
constexpr unsigned long long kSumMask = (1ULL << 55) - 1;

// Tables: one 64 KB table serves two paths, entry e of (path k, byte group) at  e * 256 + (k & 1) * 128 + group * 4
// of table k >> 1.  The kernel has no static shared memory, so its dynamic part starts at kSmemBase, right behind what the
// system reserves (checked on the host), and a look-up address is  byte << 8 | bank offset,  which ONE byte permute builds,
// plus a constant that fits the load's immediate.  (Starting the tables on a 64 KB boundary instead costs 63 KB of slack and
// sixteen registers for the table base.)
constexpr int kSmemBase = 1024;
// Two batch rows: entry e of (path k, byte group) is the pair of both rows' sums at  e * 256 + group * 8  of table k.
template <int K, int NB>
struct Tab {
    static constexpr int kBytes = (NB == 1 ? (K + 1) / 2 : K) * 65536;
    static constexpr int kTail = 256;                                 // behind the tables: the layer's descriptor and the CTA's range
    // Never so little that two CTAs share an SM: with 64 KB each the hardware put two CTAs of one launch on one SM wherever the
    // previous launch left room first, and a 4096 x 4096 layer went from 3.2 to 4.4 us.
    static constexpr int kSmem = kBytes + kTail > 116 * 1024 ? kBytes + kTail : 116 * 1024;
    __host__ __device__ static constexpr int offset(int k) { return kSmemBase + (NB == 1 ? (k >> 1) * 65536 + (k & 1) * 128 : k * 65536); }
};

template <int I, int N, typename F>
__device__ __forceinline__ void static_for(F&& f) {
    if constexpr (I < N) {
        f(std::integral_constant<int, I>{});
        static_for<I + 1, N>(f);
    }
}

struct LutLayer {
    const unsigned char* lut;
    const __half* g;
    const __half* h;
    const __half* x;
    __half* y;
    unsigned long long* acc;        // [NB][Mp], all zero between calls
    int M, N, Mp, n_rb, n_cs;
    int fix_bits;
    float inv_unit, unit, limit;    // 2^-unit_exp, 2^unit_exp, 2^fix_bits
    int pad_;                       // (keeps the size a multiple of 8)
};
static_assert(sizeof(LutLayer) % 4 == 0 && sizeof(LutLayer) <= 128, "LutLayer is copied to shared memory by one warp, a word per lane");
struct CtaRange {
    int layer, b0, b1;              // block positions [b0, b1) of that layer
};
struct LutParams {
    int n_layers;
    unsigned int* status;           // RABIT_CHECKED builds: set to 2 when an index check fails (the access is skipped)
    unsigned long long* trace;      // RABIT_TRACE builds: 8 time stamps per CTA of this launch (nullptr: none)
    LutLayer layer[kMaxGroup];
    CtaRange range[kMaxGrid];
};

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void bar_cta() { asm volatile("bar.sync 0;" ::: "memory"); }
__device__ __forceinline__ uint32_t prmt(uint32_t a, uint32_t b, uint32_t s) {
    uint32_t r;
    asm("prmt.b32 %0, %1, %2, %3;" : "=r"(r) : "r"(a), "r"(b), "r"(s));
    return r;
}
template <int OFF>
__device__ __forceinline__ float lds_f32(uint32_t addr) {
    float v;
    asm volatile("ld.shared.f32 %0, [%1+%2];" : "=f"(v) : "r"(addr), "n"(OFF));
    return v;
}
// Pairs of fp32 numbers: one look-up and one add for both batch rows.
template <int OFF>
__device__ __forceinline__ unsigned long long lds_pair(uint32_t addr) {
    unsigned long long v;
    asm volatile("ld.shared.b64 %0, [%1+%2];" : "=l"(v) : "r"(addr), "n"(OFF));
    return v;
}
__device__ __forceinline__ void add_pair(unsigned long long& sum, unsigned long long v) {
    asm("add.rn.f32x2 %0, %0, %1;" : "+l"(sum) : "l"(v));
}
__device__ __forceinline__ float2 pair_of(unsigned long long v) {
    return make_float2(__uint_as_float((uint32_t)v), __uint_as_float((uint32_t)(v >> 32)));
}
__device__ __forceinline__ void sts_f32(uint32_t addr, float v) {
    asm volatile("st.shared.f32 [%0], %1;" ::"r"(addr), "f"(v) : "memory");
}
__device__ __forceinline__ void sts_pair(uint32_t addr, float v0, float v1) {
    asm volatile("st.shared.v2.f32 [%0], {%1, %2};" ::"r"(addr), "f"(v0), "f"(v1) : "memory");
}
// Weights are read exactly once: no L1 allocation, 128-byte L2 sectors.
__device__ __forceinline__ uint4 ldg_stream(const uint4* p) {
    uint4 v;
    asm volatile("ld.global.nc.L1::no_allocate.L2::128B.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
    return v;
}
// The compiler may move an ordinary use of a loaded value up to the load and stall there; these two keep the load
// early and its first use late (volatile statements keep their order among themselves, and the look-ups are volatile).
__device__ __forceinline__ unsigned short ldg_u16_early(const unsigned short* p) {
    unsigned short v;
    asm volatile("ld.global.nc.u16 %0, [%1];" : "=h"(v) : "l"(p));
    return v;
}
__device__ __forceinline__ unsigned short use_here_u16(unsigned short v) {
    unsigned short r;
    asm volatile("mov.b16 %0, %1;" : "=h"(r) : "h"(v));
    return r;
}
__device__ __forceinline__ unsigned long long use_here_u64(unsigned long long v) {
    unsigned long long r;
    asm volatile("mov.b64 %0, %1;" : "=l"(r) : "l"(v));
    return r;
}

// Phase stamps of a CTA (RABIT_TRACE builds only; see rabit_trace_begin in rabit.h): stamp 0 is %globaltimer
// (nanoseconds, coarse) at entry, stamps 1..7 are SM clock cycles since entry, taken by lane 0 of warp 0.
#ifdef RABIT_TRACE
__device__ __forceinline__ unsigned long long global_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}
__device__ __forceinline__ unsigned long long sm_clock() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%clock64;" : "=l"(t));
    return t;
}
#define RABIT_STAMP0() do { trace_t0 = sm_clock(); if (P.trace && lane == 0 && warp == 0) P.trace[(size_t)blockIdx.x * 64] = global_ns(); } while (0)
#define RABIT_STAMP(i) do { if (P.trace && lane == 0 && warp == 0) P.trace[(size_t)blockIdx.x * 64 + (i)] = sm_clock() - trace_t0; } while (0)
#else
#define RABIT_STAMP0() do { } while (0)
#define RABIT_STAMP(i) do { } while (0)
#endif

// Checked build (-DRABIT_CHECKED, python paper_2602_05367_b200/build.py --checked): every index that addresses global or
// shared memory in this kernel is compared with its range first; a violation sets the status word to 2 and the access
// is skipped (never a trap, never an out-of-range access), so the small-shape suite can run under it in place of a
// memory checker.
#ifdef RABIT_CHECKED
#define RABIT_IN_RANGE(cond) ((cond) ? true : (atomicExch(P.status, 2u), false))
#else
#define RABIT_IN_RANGE(cond) true
#endif

template <int K>
struct Blk {
    uint4 v[2 * K];                  // one lane's 32 bytes per path: (path k, half hf) at v[2k + hf]
};
// half hf (byte groups 16 hf .. of the rotated order) of block bb of the range, every path
template <int K>
__device__ __forceinline__ void load_half(Blk<K>& r, int hf, const uint4* range_base, int bb, int lane) {
    const uint4* p = range_base + (size_t)bb * (K * RABIT_LUT_PART_BYTES / 16) + lane;
#pragma unroll
    for (int k = 0; k < K; ++k) r.v[2 * k + hf] = ldg_stream(p + (2 * k + hf) * 32);
}

// What a lane still owes for the last block it accumulated: the answer of its atomic add is looked at
// one block later, so that the round trip to L2 overlaps the next block's look-ups.
struct Pending {
    unsigned long long old, add;
    unsigned long long* word;
    bool bad, live;
};

template <int NB>
__device__ __forceinline__ void settle(Pending (&pd)[NB], const LutLayer& L) {
#pragma unroll
    for (int b = 0; b < NB; ++b) {
        if (!pd[b].live) continue;
        pd[b].live = false;
        if ((int)((pd[b].old >> 55) & 0xFFu) != L.n_cs - 1) continue;          // other slices are still to come
        const unsigned long long sum = (pd[b].old & kSumMask) + (pd[b].add & kSumMask);
        const long long total = (long long)sum - ((long long)L.n_cs << L.fix_bits);
        const bool poisoned = pd[b].bad || (pd[b].old >> 63) != 0;
        const float v = poisoned ? __int_as_float(0x7FC00000) : __ll2float_rn(total) * L.unit;
        const long long row = (pd[b].word - L.acc) - (long long)b * L.Mp;       // (rare path: the layer's fields come from shared memory)
        if (row >= 0 && row < L.M) L.y[(size_t)b * L.M + row] = __float2half_rn(v);
        *pd[b].word = 0ULL;                                                     // resting state for the next call
    }
}

template <int K, int NB>
__global__ void __launch_bounds__(kThreads, 1)
rabit_gemv_lut_kernel(const __grid_constant__ LutParams P) {
    using T = Tab<K, NB>;
    extern __shared__ __align__(1024) unsigned char smem[];             // the tables, then what the CTA needs of the launch parameters
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;

#ifdef RABIT_TRACE
    unsigned long long trace_t0;
#endif
    RABIT_STAMP0();                                                     // entry
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

    // The launch parameters live in constant memory, which is cold in every new launch: a first touch of one of its
    // lines costs a trip to L2.  Everything the CTA needs later is therefore copied to shared memory now, before the
    // dependency wait, so that none of those trips lands between the arrival of x and the end of the kernel.
    LutLayer& layer_copy = *reinterpret_cast<LutLayer*>(smem + T::kBytes);
    CtaRange& range_copy = *reinterpret_cast<CtaRange*>(smem + T::kBytes + 128);
    if (warp == 0) {
        const CtaRange r0 = P.range[blockIdx.x];
        const uint32_t* src = reinterpret_cast<const uint32_t*>(&P.layer[r0.layer]);
        if (lane < (int)(sizeof(LutLayer) / 4)) reinterpret_cast<uint32_t*>(&layer_copy)[lane] = src[lane];
        if (lane == 0) range_copy = r0;
    }
    __syncthreads();
    const CtaRange R = range_copy;
    const LutLayer& L = layer_copy;
    const int n_blocks = R.b1 - R.b0;
    const unsigned char* range_bytes = L.lut + (size_t)R.b0 * (K * RABIT_LUT_PART_BYTES);
    const uint4* range_base = reinterpret_cast<const uint4*>(range_bytes);

    // ---- everything that does not depend on the stream's past
    const int n_mine = warp < n_blocks ? (n_blocks - warp + kWarps - 1) / kWarps : 0;    // blocks warp, warp + 16, ...
    Blk<K> cur;                                          // this warp's current block
#pragma unroll
    for (int i = 0; i < 2 * K; ++i) cur.v[i] = make_uint4(0u, 0u, 0u, 0u);
    if (n_mine > 0) {
        load_half<K>(cur, 0, range_base, warp, lane);
        load_half<K>(cur, 1, range_base, warp, lane);
    }

    const uint32_t tab0 = smem_u32(smem);                // == kSmemBase
    // One row: byte q of `bank0 + 0x10101010 * j`, modulo 128: bank offset (4 * group) of the group this lane visits in step 4j + q.  A
    // permute of (weight word, that) yields byte << 8 | bank offset (its upper bytes copy a sign bit that is always clear).
    // Two rows: offsets (8 * group) take all eight bits, so the ones of steps 4j, 4j + 1 and of 4j + 2, 4j + 3 sit a halfword each, modulo 256,
    // and the permute's upper bytes are the clear byte between them.
    const uint32_t lane4 = (uint32_t)lane * 4u;
    const uint32_t bank0 = NB == 1 ? (lane4 & 127) | ((lane4 + 4) & 127) << 8 | ((lane4 + 8) & 127) << 16 | ((lane4 + 12) & 127) << 24 : ((2 * lane4) & 255) | ((2 * lane4 + 8) & 255) << 16;
    int cs = R.b0 / L.n_rb;
    int seg_rb0 = R.b0 - cs * L.n_rb;                    // row block of the first block of the current segment
    int seg_begin = 0, seg_end = min(n_blocks, L.n_rb - seg_rb0);       // blocks [seg_begin, seg_end) of the range use slice cs
    constexpr int kPairs = (8 * K + kWarps - 1) / kWarps;                // (path, upper three index bits) pairs a warp builds, 32 entries each
    uint4 hq[kPairs], xq[NB];
    auto load_h = [&](int slice) {                                      // static data: may be read before the dependency wait
#pragma unroll
        for (int u = 0; u < kPairs; ++u) {
            const int pi = warp + u * kWarps;
            const int col = slice * RABIT_LUT_COLS + 8 * lane;
            hq[u] = make_uint4(0u, 0u, 0u, 0u);
            if (pi < 8 * K && col < L.N && RABIT_IN_RANGE(slice >= 0 && slice < L.n_cs && col + 8 <= L.N)) hq[u] = __ldg(reinterpret_cast<const uint4*>(L.h + (size_t)(pi >> 3) * L.N + col));
        }
    };
    auto load_x = [&](int slice) {                                      // L2 (not L1): written by the previous kernel in the stream
        const int col = slice * RABIT_LUT_COLS + 8 * lane;
#pragma unroll
        for (int b = 0; b < NB; ++b) {
            xq[b] = make_uint4(0u, 0u, 0u, 0u);
            if (col < L.N && RABIT_IN_RANGE(slice >= 0 && slice < L.n_cs && col + 8 <= L.N)) xq[b] = __ldcg(reinterpret_cast<const uint4*>(L.x + (size_t)b * L.N + col));
        }
    };
    // table of the slice whose h and x sit in hq / xq:  entry e of (path k, group) = sum_{bit<8} (e has bit ? -t : +t),  t = h * x
    auto build_table = [&]() {
#pragma unroll
        for (int u = 0; u < kPairs; ++u) {
            const int pi = warp + u * kWarps;
            if (pi >= 8 * K) break;
            const int k = pi >> 3, ehi = pi & 7;
            const uint32_t hw[4] = {hq[u].x, hq[u].y, hq[u].z, hq[u].w};
            float v[NB][32];
#pragma unroll
            for (int b = 0; b < NB; ++b) {
                const uint32_t xw[4] = {xq[b].x, xq[b].y, xq[b].z, xq[b].w};
                float t[8];
#pragma unroll
                for (int w = 0; w < 4; ++w) {
                    const float2 hf = __half22float2(*reinterpret_cast<const __half2*>(&hw[w]));
                    const float2 xf = __half22float2(*reinterpret_cast<const __half2*>(&xw[w]));
                    t[2 * w] = hf.x * xf.x;                              // exact: two 11-bit significands
                    t[2 * w + 1] = hf.y * xf.y;
                }
                v[b][0] = (ehi & 1 ? -t[5] : t[5]) + (ehi & 2 ? -t[6] : t[6]) + (ehi & 4 ? -t[7] : t[7])
                        + (((t[0] + t[1]) + (t[2] + t[3])) + t[4]);
#pragma unroll
                for (int bit = 0; bit < 5; ++bit) {
                    const float m2 = -2.f * t[bit];
#pragma unroll
                    for (int e = 0; e < (1 << bit); ++e) v[b][e | (1 << bit)] = v[b][e] + m2;
                }
            }
            // (the start of the tables as a register or as a constant: either way round the other form loses, by allocation of registers, 28672 x 8192
            // 14.9 -> 15.3 us with one row, 20.9 -> 23.6 with two)
            const uint32_t dst = (NB == 1 ? tab0 + (k >> 1) * 65536 + (k & 1) * 128 : (uint32_t)T::offset(k)) + (ehi * 32) * 256 + lane * (4 * NB);
#pragma unroll
            for (int e = 0; e < 32; ++e)
                if (RABIT_IN_RANGE(dst + e * 256 >= tab0 && dst + e * 256 + 4 * NB <= tab0 + (uint32_t)T::kBytes)) {
                    if constexpr (NB == 1) sts_f32(dst + e * 256, v[0][e]);
                    else sts_pair(dst + e * 256, v[0][e], v[1][e]);
                }
        }
    };
    // makes the table of block bb's slice the current one; every warp crosses every slice border of the range here
    auto advance_to = [&](int bb) {
        while (bb >= seg_end) {
            bar_cta();                                                  // every warp is done with the old table
            build_table();
            cs += 1;
            seg_begin = seg_end;
            seg_rb0 = 0;
            seg_end = min(n_blocks, seg_end + L.n_rb);
            if (seg_end < n_blocks) { load_h(cs + 1); load_x(cs + 1); } // the table after this one
            bar_cta();
        }
    };
    load_h(cs);

    asm volatile("griddepcontrol.wait;" ::: "memory");
    RABIT_STAMP(1);                                                     // the previous kernel's results are visible
    if (n_blocks <= 0) return;
    load_x(cs);
#ifdef RABIT_TRACE
    if (xq[0].x == 0x12345678u && xq[0].y == 0x9ABCDEF0u && hq[0].x == 0x12345678u) RABIT_STAMP(7);   // (a use of x and h, so that the next stamp follows their arrival)
#endif
    RABIT_STAMP(2);                                                     // x and h of the first table have arrived
    build_table();
    if (seg_end < n_blocks) { load_h(cs + 1); load_x(cs + 1); }
    bar_cta();
    RABIT_STAMP(3);                                                     // first table built

    // One iteration per block of this warp.  This block's output scales and the atomic adds of the previous block are ISSUED at the
    // top of an iteration and their results first touched below its look-ups, some 1300 cycles later; the next block's weights
    // set off when the look-ups have used up the registers they go to.
    // what every iteration needs of the layer, in registers (the shared-memory pipe is the one this loop saturates)
    const unsigned short* const g_base = reinterpret_cast<const unsigned short*>(L.g);
    unsigned long long* const acc_base = L.acc;
    const int Mp = L.Mp;
    const float inv_unit = L.inv_unit, limit = L.limit;
    const long long bias = (1LL << L.fix_bits) + (1LL << 55);            // shift to non-negative + one arrival
    Pending pd[NB];
#pragma unroll
    for (int b = 0; b < NB; ++b) { pd[b].live = false; pd[b].old = 0ULL; pd[b].add = 0ULL; pd[b].word = nullptr; pd[b].bad = false; }
    bool owe = false;                                                   // pd holds a finished block whose atomics are still to be issued
    for (int i = 0; i < n_mine; ++i) {
        const int bb = warp + i * kWarps;
#ifdef RABIT_TRACE
        if (i < 11) RABIT_STAMP(8 + 5 * i);                             // iteration i: top
#endif
        advance_to(bb);
        const int row = (seg_rb0 + (bb - seg_begin)) * RABIT_LUT_ROWS + lane;
        unsigned short graw[K];
#pragma unroll
        for (int k = 0; k < K; ++k) {
            graw[k] = 0;
            if (RABIT_IN_RANGE(row >= 0 && row < Mp)) graw[k] = ldg_u16_early(g_base + (size_t)k * Mp + row);
        }
        const int bb_next = bb + kWarps;
        const bool next_ok = i + 1 < n_mine && RABIT_IN_RANGE(bb_next >= 0 && bb_next < n_blocks && (long long)R.b0 + bb_next < (long long)L.n_cs * L.n_rb);
        if (owe) {
#pragma unroll
            for (int b = 0; b < NB; ++b) {
                if (!RABIT_IN_RANGE(pd[b].word >= acc_base && pd[b].word < acc_base + (size_t)NB * Mp)) continue;
                if (pd[b].bad) atomicOr(pd[b].word, 1ULL << 63);
                pd[b].old = atomicAdd(pd[b].word, pd[b].add);
                pd[b].live = true;
            }
        }
        if (i == 0) RABIT_STAMP(4);                                     // first weights in registers
#ifdef RABIT_TRACE
        {
            unsigned int u = cur.v[0].x;
#pragma unroll
            for (int t = 0; t < 2 * K; ++t) u |= cur.v[t].w;
            u = (unsigned int)use_here_u64(u);                           // the block's weights have arrived
            if (i < 11 && u != 0x13572468u) RABIT_STAMP(9 + 5 * i);
        }
#endif

        // sums of the even and the odd byte groups, two rows' as pairs
        std::conditional_t<NB == 1, float, unsigned long long> acc[K][2];
#pragma unroll
        for (int k = 0; k < K; ++k) acc[k][0] = acc[k][1] = 0;
        constexpr bool kAhead = NB > 1 && K < 3;                        // (three paths: 24 registers that there are not, 22016 x 4096 16.1 instead of 15.2 us)
        // The next block's weights.  One row: into the registers that the look-ups have used up, all together behind the last of them: the
        // other warps' look-ups cover the wait (into registers of their own behind the first step 28672 x 8192 15.0 -> 16.8 us).  Two rows, whose
        // look-ups take longer than the wait: into registers of their own behind the first of the eight steps (28672 x 8192 20.9 us; behind the
        // second 21.9, the fourth 24.5, the last 24.1; above this block's scales and atomics 21.4).
        [[maybe_unused]] Blk<!kAhead ? 1 : K> ahead;
        if constexpr (kAhead) ahead = cur;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const uint32_t bank = NB == 1 ? (bank0 + 0x10101010u * (uint32_t)j) & 0x7F7F7F7Fu : (bank0 + 0x00200020u * (uint32_t)j) & 0x00F800F8u;
            const uint32_t bank2 = (bank0 + 0x00200020u * (uint32_t)j + 0x00100010u) & 0x00F800F8u;
            static_for<0, K>([&](auto kc) {
                constexpr int k = decltype(kc)::value;
                const uint4 part = cur.v[2 * k + (j >> 2)];
                const uint32_t w = (j & 3) == 0 ? part.x : (j & 3) == 1 ? part.y : (j & 3) == 2 ? part.z : part.w;
                // sign byte << 8 | bank offset, from one permute
                const uint32_t a0 = prmt(w, bank, NB == 1 ? 0xCC04 : 0x5504), a1 = prmt(w, bank, NB == 1 ? 0xCC15 : 0x5516);
                const uint32_t a2 = prmt(w, NB == 1 ? bank : bank2, NB == 1 ? 0xCC26 : 0x5524), a3 = prmt(w, NB == 1 ? bank : bank2, NB == 1 ? 0xCC37 : 0x5536);
#ifdef RABIT_CHECKED
                {
                    const uint32_t hi = NB == 1 ? 65536u - 128u : 65536u;   // with the path offset added: inside its table
                    if (!RABIT_IN_RANGE(a0 < hi && a1 < hi && a2 < hi && a3 < hi)) return;
                }
#endif
                if constexpr (NB == 1) {
                    acc[k][0] += lds_f32<T::offset(k)>(a0);
                    acc[k][1] += lds_f32<T::offset(k)>(a1);
                    acc[k][0] += lds_f32<T::offset(k)>(a2);
                    acc[k][1] += lds_f32<T::offset(k)>(a3);
                } else {
                    const unsigned long long v0 = lds_pair<T::offset(k)>(a0), v1 = lds_pair<T::offset(k)>(a1), v2 = lds_pair<T::offset(k)>(a2), v3 = lds_pair<T::offset(k)>(a3);
                    add_pair(acc[k][0], v0);
                    add_pair(acc[k][1], v1);
                    add_pair(acc[k][0], v2);
                    add_pair(acc[k][1], v3);
                }
            });
            if (j == (!kAhead ? 7 : 0) && next_ok) {
                if constexpr (!kAhead) { load_half<K>(cur, 0, range_base, bb_next, lane); load_half<K>(cur, 1, range_base, bb_next, lane); }
                else { load_half<K>(ahead, 0, range_base, bb_next, lane); load_half<K>(ahead, 1, range_base, bb_next, lane); }
            }
        }
        if constexpr (kAhead) cur = ahead;
#ifdef RABIT_TRACE
        if (i == 0) RABIT_STAMP(7);                                     // first block's look-ups issued
        if (i < 11 && use_here_u64((unsigned long long)(acc[0][0] + acc[0][1] + acc[K - 1][0] + acc[K - 1][1])) != 0x13572468u) RABIT_STAMP(10 + 5 * i);   // look-ups answered
#endif
#pragma unroll
        for (int b = 0; b < NB; ++b) pd[b].old = use_here_u64(pd[b].old);
        settle<NB>(pd, L);                                               // the previous block's atomics, issued above the look-ups
#ifdef RABIT_TRACE
        if (i < 11) RABIT_STAMP(11 + 5 * i);                            // previous atomic answered and settled
#endif
#pragma unroll
        for (int k = 0; k < K; ++k) graw[k] = use_here_u16(graw[k]);
#ifdef RABIT_TRACE
        if (i < 11) RABIT_STAMP(12 + 5 * i);                            // output scales have arrived
#endif
#pragma unroll
        for (int b = 0; b < NB; ++b) {
            float p = 0.f;
#pragma unroll
            for (int k = 0; k < K; ++k) {
                float sum;
                if constexpr (NB == 1) {
                    sum = acc[k][0] + acc[k][1];
                } else {
                    const float2 even = pair_of(acc[k][0]), odd = pair_of(acc[k][1]);
                    sum = b == 0 ? even.x + odd.x : even.y + odd.y;
                }
                p += __half2float(__ushort_as_half(graw[k])) * sum;
            }
            const float scaled = p * inv_unit;
            const bool bad = !(fabsf(scaled) < limit);                    // inf or NaN: finite inputs cannot get here
            const long long qv = bad ? 0LL : __float2ll_rn(scaled);
            pd[b].add = (unsigned long long)(qv + bias);
            pd[b].word = acc_base + (size_t)b * Mp + row;
            pd[b].bad = bad;
        }
        owe = true;
    }
    if (owe) {
#pragma unroll
        for (int b = 0; b < NB; ++b) {
            if (!RABIT_IN_RANGE(pd[b].word >= acc_base && pd[b].word < acc_base + (size_t)NB * Mp)) continue;
            if (pd[b].bad) atomicOr(pd[b].word, 1ULL << 63);
            pd[b].old = atomicAdd(pd[b].word, pd[b].add);
            pd[b].live = true;
        }
    }
    RABIT_STAMP(5);                                                     // last look-up done, last atomic issued
    advance_to(n_blocks - 1);                                           // warps that ran out of blocks early still take part in the rebuilds
    settle<NB>(pd, L);
    RABIT_STAMP(6);                                                     // last atomic answered, y stored
}

// ---- host side: cutting the layers into ranges of equal cost ------------------------------------

struct Cost {
    long long block, table;
};
// A block of K paths (look-ups, loads, its atomic) and a table (build plus the two barriers around it); only their ratio matters
// for the cut.  (The block's figure is in clocks of an earlier loop: it takes 118 now.)
// (the table figure is a fit: the split that minimises the measured step time charges a table about 26 blocks, far
// more than its 430 cycles of stores, because a rebuild in mid-range also stops every warp at two barriers)
// (two batch rows: a quarter less measures best; 22016 x 4096 10.2, 9.9, 9.85 us and 28672 x 8192 20.9, 20.9, 21.3 with 1900, 1700, 1500;
// of three paths 5000 x 13824 14.35, 14.15, 12.95, 22016 x 4096 15.2, 15.2, 14.8, 28672 x 8192 32.05, 32.0, 32.2 with 2400, 1700, 1200)
Cost cost_of(int K, int nb) { return Cost{(long long)nb * (70 * K + 30), (long long)nb * ((nb == 1 ? 2200 : K == 3 ? 1200 : 1700) * K) + 100}; }

// CTAs a layer of n_cs x n_rb blocks needs when no CTA may cost more than `limit`; writes the cuts if asked.
int ctas_needed(int n_cs, int n_rb, const Cost& C, long long limit, std::vector<int>* cuts) {
    const long long total = (long long)n_cs * n_rb;
    long long pos = 0;
    int n = 0;
    if (cuts) { cuts->clear(); cuts->push_back(0); }
    while (pos < total) {
        long long budget = limit, taken = 0;
        long long p = pos;
        while (p < total) {
            budget -= C.table;
            const long long can = budget / C.block;
            if (can < 1) break;
            const long long left_in_slice = n_rb - (p % n_rb);
            const long long take = std::min(can, left_in_slice);
            p += take; taken += take; budget -= take * C.block;
            if (take < left_in_slice) break;
        }
        if (taken == 0) return 1 << 30;                                  // the limit does not even pay for one block
        pos = p;
        ++n;
        if (cuts) cuts->push_back((int)pos);
        if (n > (1 << 20)) return 1 << 30;
    }
    return n;
}

// Smallest per-CTA cost with which the layer fits into n_cta CTAs.
long long best_limit(int n_cs, int n_rb, const Cost& C, int n_cta) {
    long long lo = C.table + C.block, hi = (long long)n_cs * (C.table + (long long)n_rb * C.block);
    while (lo < hi) {
        const long long mid = (lo + hi) / 2;
        if (ctas_needed(n_cs, n_rb, C, mid, nullptr) <= n_cta) hi = mid; else lo = mid + 1;
    }
    return lo;
}

template <int K, int NB>
cudaError_t launch_inst(const LutParams& P, int grid, int device, cudaStream_t stream) {
    static bool attr_done[64] = {false};
    const size_t smem = (size_t)Tab<K, NB>::kSmem;
    if (device < 0 || device >= 64 || !attr_done[device]) {
        cudaError_t e = cudaFuncSetAttribute(rabit_gemv_lut_kernel<K, NB>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        if (device >= 0 && device < 64) attr_done[device] = true;
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
    return cudaLaunchKernelEx(&cfg, rabit_gemv_lut_kernel<K, NB>, P);
}

cudaError_t launch_k(int K, int batch, const LutParams& P, int grid, int device, cudaStream_t stream) {
    if (K == 1) return batch == 1 ? launch_inst<1, 1>(P, grid, device, stream) : launch_inst<1, 2>(P, grid, device, stream);
    if (K == 2) return batch == 1 ? launch_inst<2, 1>(P, grid, device, stream) : launch_inst<2, 2>(P, grid, device, stream);
    return batch == 1 ? launch_inst<3, 1>(P, grid, device, stream) : launch_inst<3, 2>(P, grid, device, stream);
}

}  // namespace

int rabit_gemv_lut_max_rows() { return 2; }

// whether dynamic shared memory starts where the look-up addresses assume it
static bool smem_base_ok(int device) {
    static signed char known[64] = {0};                                  // 0 not asked yet, 1 yes, -1 no
    signed char* k = device >= 0 && device < 64 ? &known[device] : nullptr;
    if (k && *k) return *k > 0;
    int reserved = -1;
    const bool ok = cudaDeviceGetAttribute(&reserved, cudaDevAttrReservedSharedMemoryPerBlock, device) == cudaSuccess && reserved == kSmemBase;
    if (k) *k = ok ? 1 : -1;
    return ok;
}

bool rabit_gemv_lut_supports(const rabit_layer& L, int batch) {
    if (batch < 1 || batch > 2 || !smem_base_ok(L.device)) return false;
    if (L.geom.n_cs > RABIT_LUT_MAX_SLICES) return false;
    return (long long)L.geom.n_cs * L.geom.n_rb < (1LL << 30) && L.d_lut != nullptr && L.d_acc != nullptr;
}

// Whether it is the faster one for layers that it can run.  Against the f16 GEMV only two rows of three paths are ever not: its tables take
// a table's build (three of 64 KB) per CTA and pay from about four blocks of 32 rows x 256 columns per SM on (B200, us, f16 GEMV against this:
// 2000 x 1024 (256 blocks) 3.67 / 4.1, 2048 x 2048 (512) 4.1 / 4.2, 1024 x 4096 (512) 4.1 / 4.0, 11008 x 512 (688) 5.0 / 4.6, 2048 x 3072 (768)
// 5.0 / 4.3, 4096 x 4096 7.4 / 5.7, 22016 x 4096 24.2 / 14.8, 28672 x 8192 54.0 / 32.0).
bool rabit_gemv_lut_preferred(const rabit_layer* const* layers, int n_layers, int batch) {
    if (layers[0]->geom.K < 3 || batch == 1) return true;
    long long blocks = 0;
    for (int l = 0; l < n_layers; ++l) blocks += (long long)layers[l]->geom.n_cs * layers[l]->geom.n_rb;
    return blocks > 4LL * (layers[0]->sm_count > 0 ? layers[0]->sm_count : 148);
}

bool rabit_gemv_lut_group_supports(const rabit_layer* const* layers, int n_layers, int batch) {
    if (n_layers < 1 || n_layers > kMaxGroup) return false;
    for (int l = 0; l < n_layers; ++l) {
        if (!rabit_gemv_lut_supports(*layers[l], batch) || layers[l]->geom.K != layers[0]->geom.K) return false;
        for (int m = 0; m < l; ++m)
            if (layers[m] == layers[l]) return false;                    // one layer twice would share its accumulate words
    }
    return true;
}

// One launch for n_layers independent layers of equal K and 1..2 batch rows (x_l: [batch][N_l], y_l: [batch][M_l]).
cudaError_t rabit_launch_gemv_lut_group(const rabit_layer* const* layers, int n_layers, const void* const* xs, void* const* ys,
                                        int batch, cudaStream_t stream, unsigned long long* const* acc_override, unsigned int* status_override) {
    if (!rabit_gemv_lut_group_supports(layers, n_layers, batch)) return cudaErrorInvalidValue;
    const int K = layers[0]->geom.K;
    LutParams P;
    P.n_layers = n_layers;
    P.status = status_override ? status_override : layers[0]->d_status;  // (only a checked build writes it: this kernel has no wait that could run out)
    P.trace = nullptr;
    const Cost C = cost_of(K, batch);
    long long weight[kMaxGroup], total_weight = 0, total_blocks = 0;
    for (int l = 0; l < n_layers; ++l) {
        const rabit_layer& Ly = *layers[l];
        const RabitGeom& G = Ly.geom;
        LutLayer& D = P.layer[l];
        D.lut = Ly.d_lut;
        D.g = (const __half*)Ly.d_g;
        D.h = (const __half*)Ly.d_h;
        D.x = (const __half*)xs[l];
        D.y = (__half*)ys[l];
        D.acc = acc_override ? acc_override[l] : Ly.d_acc;
        D.M = G.M; D.N = G.N; D.Mp = G.Mp; D.n_rb = G.n_rb; D.n_cs = G.n_cs;
        D.fix_bits = G.fix_bits;
        D.unit = ldexpf(1.f, G.unit_exp);
        D.inv_unit = ldexpf(1.f, -G.unit_exp);
        D.limit = ldexpf(1.f, G.fix_bits);
        const long long blocks = (long long)G.n_cs * G.n_rb;
        weight[l] = blocks * C.block + (long long)G.n_cs * C.table;
        total_weight += weight[l];
        total_blocks += blocks;
    }
    for (int l = n_layers; l < kMaxGroup; ++l) P.layer[l] = P.layer[0];
    // The cut of the layers into ranges depends only on the shapes, the batch and the device: remembered per thread
    // (a decoder calls the same few groups over and over; the search costs a few microseconds of host time).
    struct PlanKey { int n, batch, sms, shape[kMaxGroup][3]; };
    struct Plan { PlanKey key; int grid; CtaRange range[kMaxGrid]; };
    static thread_local std::vector<Plan> plans;
    PlanKey key;
    std::memset(&key, 0, sizeof(key));
    key.n = n_layers; key.batch = batch; key.sms = layers[0]->sm_count;
    for (int l = 0; l < n_layers; ++l) { key.shape[l][0] = K; key.shape[l][1] = layers[l]->geom.n_rb; key.shape[l][2] = layers[l]->geom.n_cs; }
    for (const Plan& pl : plans)
        if (std::memcmp(&pl.key, &key, sizeof(key)) == 0) {
            std::memcpy(P.range, pl.range, sizeof(P.range));
            P.trace = rabit_trace_slot(pl.grid);
            return launch_k(K, batch, P, pl.grid, layers[0]->device, stream);
        }
    int sms = layers[0]->sm_count > 0 ? layers[0]->sm_count : 148;
    int grid = sms < kMaxGrid ? sms : kMaxGrid;
    if ((long long)grid > total_blocks) grid = (int)total_blocks;
    if (grid < n_layers) grid = n_layers;                                // (n_layers <= 8 <= any device's SM count)

    // share the CTAs out in proportion to the cost, at least one each, then move single CTAs from the
    // layer that finishes first to the one that finishes last while that lowers the finishing time
    int n_cta[kMaxGroup], given = 0;
    for (int l = 0; l < n_layers; ++l) {
        long long n = (long long)grid * weight[l] / total_weight;
        const long long blocks = (long long)layers[l]->geom.n_cs * layers[l]->geom.n_rb;
        if (n < 1) n = 1;
        if (n > blocks) n = blocks;
        n_cta[l] = (int)n;
        given += n_cta[l];
    }
    auto blocks_of = [&](int l) { return (long long)layers[l]->geom.n_cs * layers[l]->geom.n_rb; };
    while (given > grid) {
        int best = -1;
        for (int l = 0; l < n_layers; ++l)
            if (n_cta[l] > 1 && (best < 0 || weight[l] * n_cta[best] < weight[best] * n_cta[l])) best = l;
        if (best < 0) break;
        n_cta[best] -= 1; given -= 1;
    }
    while (given < grid) {
        int best = -1;
        for (int l = 0; l < n_layers; ++l)
            if (n_cta[l] < blocks_of(l) && (best < 0 || weight[l] * n_cta[best] > weight[best] * n_cta[l])) best = l;
        if (best < 0) break;
        n_cta[best] += 1; given += 1;
    }
    long long limit[kMaxGroup];
    for (int l = 0; l < n_layers; ++l) limit[l] = best_limit(layers[l]->geom.n_cs, layers[l]->geom.n_rb, C, n_cta[l]);
    for (int iter = 0; iter < 8 && n_layers > 1; ++iter) {
        int hi = 0, lo = 0;
        for (int l = 1; l < n_layers; ++l) {
            if (limit[l] > limit[hi]) hi = l;
            if (limit[l] < limit[lo]) lo = l;
        }
        if (hi == lo || n_cta[lo] <= 1 || n_cta[hi] >= blocks_of(hi)) break;
        const long long lo_new = best_limit(layers[lo]->geom.n_cs, layers[lo]->geom.n_rb, C, n_cta[lo] - 1);
        const long long hi_new = best_limit(layers[hi]->geom.n_cs, layers[hi]->geom.n_rb, C, n_cta[hi] + 1);
        if (std::max(lo_new, hi_new) >= limit[hi]) break;
        n_cta[lo] -= 1; n_cta[hi] += 1;
        limit[lo] = lo_new; limit[hi] = hi_new;
    }
    int c0 = 0;
    std::vector<int> cuts;
    for (int l = 0; l < n_layers; ++l) {
        const int used = ctas_needed(layers[l]->geom.n_cs, layers[l]->geom.n_rb, C, limit[l], &cuts);
        if (used > n_cta[l] || c0 + used > kMaxGrid) return cudaErrorInvalidValue;      // cannot happen: limit[l] was found with n_cta[l]
        for (int i = 0; i < used; ++i) {
            P.range[c0 + i] = CtaRange{l, cuts[i], cuts[i + 1]};
        }
        c0 += used;
    }
    const int launch_grid = c0;
    for (int i = c0; i < kMaxGrid; ++i) P.range[i] = CtaRange{0, 0, 0};
    if (plans.size() >= 256) plans.clear();
    plans.emplace_back();
    plans.back().key = key;
    plans.back().grid = launch_grid;
    std::memcpy(plans.back().range, P.range, sizeof(P.range));
    P.trace = rabit_trace_slot(launch_grid);
    return launch_k(K, batch, P, launch_grid, layers[0]->device, stream);
}

cudaError_t rabit_launch_gemv_lut(const rabit_layer& L, const void* x, void* y, int batch, cudaStream_t stream) {
    const rabit_layer* one = &L;
    return rabit_launch_gemv_lut_group(&one, 1, &x, &y, batch, stream, nullptr, nullptr);
}
