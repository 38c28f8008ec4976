// The layer on the tcgen05 tensor cores (batch > 8).
//
//   y[b][i] = sum_k g_k[i] * sum_j (B_k[i][j] * h_k[j]) * x[b][j]                       (Section 4.1, Eq. 2)
//
// For many activation rows the layer is a dense contraction.  Per path k the A operand is the sign tile with the input
// scale folded in, A_k[i][j] = +-h_k[j]: an fp16 value with its sign bit flipped by the weight bit, so the expansion is
// exact.  The B operand is x itself (fp16, loaded by TMA, shared by all paths), products are exact in fp32 and
// accumulate in fp32 in tensor memory; the epilogue applies g_k, adds the paths and rounds once to fp16.
//
// A lives in TENSOR MEMORY.  The expander warps write +-h straight from registers with tcgen05.st and the MMAs read it
// there, so the expanded operand (16 bits per weight and path) crosses shared memory neither on its way in nor out.
// Measured on B200: an M = 128, K = 16 MMA with N batch columns takes N/2 clocks all the way down to N = 16 (9.2) with A in
// tensor memory, and stores to tensor memory from other warps do not slow it; with A in shared memory N/2 only down to
// N = 128, then 32 + N/4 (its 4 KB through the shared-memory port).  Both figures need the issuing warp to be converged (one
// elected lane of a uniform loop): from a divergent single thread an MMA costs 90 to 125 clocks of issue whatever its N.
//
// Warps of a CTA:
//   0      producer: per one to four 64-column steps the x rows by TMA (128-byte swizzle) into one ring, per eight steps the packed sign
//          tiles and the h slices of every path by bulk copies into another; the first weights set off before the
//          dependency wait.  (Few, large copies: with one per step and path, and x in boxes of 16 rows, this warp was
//          what the CTA waited for: 28672 x 8192 at batch 512 390 us with boxes of 16 rows, 350 with two boxes a step.)
//   1..3   warp 1 allocates tensor memory; each issues the MMAs of the units of one accumulator and commits units and stages
//          back (a unit is a step of one path; one path uses up to four accumulators in turn, added in the epilogue).
//          One issuing warp took about 430 clocks per unit, mostly its own waits, where the four MMAs need 2 N.
//   4..19  expanders: four warpgroups (three if there are three paths) take the units in turn; warp q of a group owns
//          tensor-memory lanes 32q..32q+31, i.e. the row blocks p = 2q, 2q + 1 of a sign tile.  tcgen05.st.16x256b takes a
//          warp's registers in the same arrangement in which the tile keeps them (lane (gq, tq): rows gq, gq + 8, four
//          consecutive columns at 4 tq): a mask and a multiplication (in place of a shift) per word, then per two operand
//          registers a byte permute, a logic instruction and a fused multiply-add.  Then (same warps) the epilogue: tcgen05.ld, g_k, sum of the paths, fp16,
//          store.
//   then   the fourth issuing warp, where there is one; in stream kernels four warps for the epilogue of every pass but a task's last.
//
// Work.  One CTA per SM.  An output tile is 128 weight rows x N batch columns, N a multiple of 16 chosen for the call.
// Up to 16 batch columns a CTA takes a contiguous range of (row tile, slice of 256 columns) pairs and the parts of a row tile meet in
// its accumulate words (stream_plan; the stream kernels, NL > 1, up to four layers in a launch).  Otherwise make_plan() picks between: whole tiles;
// tiles whose contraction is split over a cluster of 2 to 8 CTAs that add their partial results through distributed shared
// memory (fixed order, no atomics); and, for long batches, contiguous ranges of 16-column groups in (row tile, group) order,
// one per SM, so that no last wave is left over.
//
// What bounds it (B200): a unit takes the larger of its four MMAs (32 clocks per 16 batch columns, and 52) and the expansion,
// 172 clocks at 16 columns (28672 x 8192).  The expansion's 20 operations of the ALU pipe per tile and warp are 80 of them; without the
// arithmetic a unit takes 143, without the MMAs 147, without stores 163, with none of the three 92: hand-overs between the roles (a wait
// on a barrier takes some 100 clocks even if it need not wait) and all of them together, no single one.  Tried without gain: three units'
// room per group (no faster), handing a unit over later so that the next one's loads come first (5 % slower).  A launch has 4 to 5 us beside
// its units: of a 4096 x 4096 launch at 16 rows, in clocks of a median CTA, 3300 from the end of the dependency wait to the first MMA (tensor memory 800,
// first weights seen 1300, x 820, first unit 370) and 3000 from the last MMA to the exit (sums and the atomics' answers 2260,
// teardown 700).  14336 x 4096 at batch 48 16.3 -> 15.8 us, 28672 x 8192 at 16 43.5 -> 41.2 (28 operations a tile before) -> 40.2 (epilogues beside), 5000 x 13824 with three paths at 200 209 -> 80
// under sustained load, when the power cap sets the clock (68 to 70 alone).
//
// Every wait on a barrier of shared memory is bounded.  On a time-out the CTA skips its remaining waits and the producer starts no
// further copy; the other roles run on (an MMA on the wrong operand is harmless, and taking the accumulate words through their
// full count leaves them at rest).  Copies and MMAs under way are awaited, again with a limit, before the tensor memory is freed,
// the status word is set and the CTA returns.  (tcgen05.alloc and the cluster barriers have no bounded form.  The first ends
// because no two CTAs of this kernel share an SM, see fill_resources, and waits for a foreign one's to leave; the second
// because every thread reaches them after bounded waits.)  DEQ (rabit_set_variant 4): the expander forms the dequantised weight sum_k +-g_k h_k in fp16 and one
// contraction serves all paths (a K-th of the tensor work, one fp16 rounding per partial product and weight).
#include <cuda.h>
#include <cuda_fp16.h>

#include <algorithm>
#include <cstddef>
#include <type_traits>
#include <vector>

#include "rabit_internal.h"
#include "rabit_tcgen05.h"

namespace {

using namespace rabit_tc;

constexpr int kTileM = 128;                 // weight rows per output tile
constexpr int kStepCols = 64;               // input columns per pipeline step (128 bytes of fp16: one swizzle row)
constexpr int kGroupCols = 16;              // batch columns come in groups of 16 (MMA N granularity)
constexpr int kUnitCols = kStepCols / 2;    // tensor-memory columns of one expanded unit (128 rows x 64 columns of fp16)
constexpr int kMaxStages = 8, kMaxUnits = 8;
constexpr int kSliceSteps = RABIT_LUT_COLS / kStepCols;   // steps of a 256-column slice
constexpr int kWSteps = 8;                  // steps per stage of the weight ring
constexpr int kWTiles = 2 * kWSteps, kWBytes = kWTiles * (RABIT_TILE_BYTES + RABIT_TILE_COLS * 2);   // per path
constexpr int kMaxWStages = 4;
constexpr int kExpandGroups = 4;            // of four warps each
constexpr int kExpandWarps = 4 * kExpandGroups;
constexpr int kFourthIssuer = 4 + kExpandWarps;
constexpr int kMaxAcc = 4;                  // accumulators
// Most accumulators of an instance.  The dequantised form of several paths, one operand per step too, has two: its expanders have more to do for
// a step than an issuing warp (with four, two paths 14336 x 4096 at 40 rows 16.5 -> 17.0 us).
__host__ __device__ constexpr int most_acc(int K, bool deq, bool seq) { return seq ? 1 : !deq ? (K == 1 ? kMaxAcc : K) : K == 1 ? kMaxAcc : 2; }
// Threads of an instance: a fourth issuing warp if there may be four accumulators, in stream kernels four warps for the epilogues.
__host__ __device__ constexpr int threads_of(int K, bool deq, bool seq, bool stream) { return (kFourthIssuer + (most_acc(K, deq, seq) > 3 ? 1 : 0) + (stream ? 4 : 0)) * 32; }
constexpr unsigned long long kSumMask = (1ULL << 55) - 1;

constexpr int kMaxTasks = 512;
constexpr long long kMaxPairs = 1LL << 23; // (row tile, slice) pairs of a stream launch
constexpr int kMaxGroup = 4;                // layers of a grouped launch

struct GemmLayer {
    const unsigned char* bits;
    const __half* g;
    const __half* h;
    __half* y;
    unsigned int* status;
    unsigned long long* acc;                // stream: accumulate words [16][Mp], all zero between calls, and their grid
    int M, N, Mp, n_rt, n_ct, n_cs;
    int fix_bits;
    float inv_unit, unit, limit;
    int pair0;                              // grouped launch: (row tile, slice) pairs of the layers before this one
};
template <int NL>
struct GemmParams {
    int n_layers;
    int batch;
    int n16;                                // groups of 16 batch columns
    int n_tasks;                            // tasks of the grid: one per CTA, or one per cluster if split > 1
    int chunks, chunk16;                    // > 0: a task is (row tile, chunk of chunk16 groups); 0: a contiguous range of groups
    int n_groups, quot, rem;                // row tiles * n16 (stream kernels, NL > 1: row tiles * n_cs, over all layers); that by n_tasks
    int max16;                              // most groups one pass can accumulate
    int split;                              // CTAs (one cluster) that share the contraction of a task, up to 8
    int recv_off;                           // receive buffer of a split task, from the control block
    int stages, stage_bytes, x_steps;       // x ring: bytes and steps of one stage
    int w_stages;                           // weight ring, behind the x ring: per stage the sign tiles [K][8][512], then h [K][256]
    int box16;                              // groups of 16 batch columns per TMA box
    int n_acc;                              // accumulators (and issuing warps)
    int paths;                              // path-major tasks: how many
    int units, a_col;                       // expanded-unit ring in tensor memory: unit u % units at columns a_col + 32 * that
#ifdef RABIT_CHECKED
    int withhold;                           // x stage before which the producer waits for a barrier that nobody signals; -1: none
#endif
    GemmLayer L[NL];
};
template <int NL>
struct alignas(64) XMaps {
    CUtensorMap map[NL];
};

struct Control {                            // ahead of the ring in shared memory
    unsigned long long full[kMaxStages];    // x of the stage landed
    unsigned long long empty[kMaxStages];   // MMAs that read it retired
    unsigned long long w_full[kMaxWStages]; // weights of the stage landed
    unsigned long long w_empty[kMaxWStages];// every expander warp has read them
    unsigned long long a_ready[kMaxUnits];  // unit expanded
    unsigned long long a_empty[kMaxUnits];  // MMAs that read the unit retired
    unsigned long long acc_ready[3];        // all MMAs of the pass retired (which one: ready_of)
    unsigned long long acc_empty[2];        // epilogue has read the accumulators
    unsigned long long drained[kMaxAcc];          // after a time-out: everything this accumulator's warp issued has retired
#ifdef RABIT_CHECKED
    unsigned long long never;               // nothing arrives here (rabit_selftest_withhold)
#endif
    uint32_t tmem_base;
    int abort_flag;
    int x_begun, w_begun;                   // stages the producer started copies for, once it has left its loop; -1 before
};
constexpr int kControlBytes = 1024;
static_assert(sizeof(Control) <= kControlBytes, "control block");

// Checked build (-DRABIT_CHECKED, python paper_2602_05367_b200/build.py --checked): every index that addresses global, shared or
// tensor memory is compared with its range first; a violation sets the status word to 2 and the access is skipped (never a
// trap; roles that wait for a skipped one end by their time-out).  In the ordinary build the checks compile to nothing.
#ifdef RABIT_CHECKED
#define RABIT_IN_RANGE(cond) ((cond) ? true : (atomicExch(P.L[0].status, 2u), false))
__device__ __forceinline__ uint32_t smem_bytes() {
    uint32_t v;
    asm volatile("mov.u32 %0, %%dynamic_smem_size;" : "=r"(v));
    return v;
}
#else
#define RABIT_IN_RANGE(cond) true
#endif

// One role's walk through a ring: every `stride`-th slot, with the parity of the slot's current lap.  A ring is a multiple of
// every stride in use, so a slot is met by the same warps in every lap and a warp that waits for a slot's barrier is
// never two laps from it (the parity would not tell the two apart).
struct Walk {
    int slot;
    uint32_t lap = 0;
    __device__ __forceinline__ void step(int stride, int size) {
        slot += stride;
        if (slot >= size) { slot -= size; lap ^= 1u; }
    }
};

// a * m on the multiply-add pipe
__device__ __forceinline__ uint32_t mul_lo(uint32_t a, uint32_t m) {
    uint32_t r;
    asm("mul.lo.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(m));
    return r;
}
struct TileIn {                             // a lane's words of a sign tile and the input scales of its columns
    uint4 w;
    uint2 h[2];
};

// A task's passes: runs of groups inside one row tile, at most max16 groups each, cut evenly.
struct Pass {
    int l, rt, c16, n;                      // layer, row tile, first group, groups
    int s_lo, s_hi;                         // steps
    int path;                               // path-major tasks: of this pass
};
template <int NL, bool SEQ>
struct PassWalker {
    int l, rt, c16, left;                   // where the next pass starts, groups left in the task (stream: slice and slices)
    int s_lo, s_hi;
    int path = 0;
    // rank: which part of the steps (split contraction)
    __host__ __device__ PassWalker(const GemmParams<NL>& P, int task, int rank) {
        l = 0;
        if (NL == 1) {
            const int n_steps = (P.L[0].N + kStepCols - 1) / kStepCols;   // N % 32 == 0: the last step may hold one column tile only
            s_lo = (int)((long long)n_steps * rank / P.split);
            s_hi = (int)((long long)n_steps * (rank + 1) / P.split);
        }
        if (NL == 1 && P.chunks > 0) {
            rt = task / P.chunks;
            c16 = (task - rt * P.chunks) * P.chunk16;
            left = min(P.chunk16, P.n16 - c16);
        } else {
            // floor(n_groups * task / n_tasks), from quotient and remainder of n_groups: no 64-bit division
            int g = P.quot * task + P.rem * task / P.n_tasks;
            left = P.quot * (task + 1) + P.rem * (task + 1) / P.n_tasks - g;
            if (NL > 1) {
                while (l + 1 < P.n_layers && g >= P.L[l + 1].pair0) ++l;
                g -= P.L[l].pair0;
            }
            const int per_rt = NL > 1 ? P.L[l].n_cs : P.n16;
            rt = g / per_rt;
            c16 = g - rt * per_rt;
        }
    }
    __host__ __device__ bool next(const GemmParams<NL>& P, Pass& ps) {
        if (left <= 0) return false;
        if (NL > 1) {
            const int n_cs = P.L[l].n_cs, run = min(left, n_cs - c16);
            ps = Pass{l, rt, 0, 1, c16 * kSliceSteps, min((c16 + run) * kSliceSteps, (P.L[l].n_ct + 1) / 2), 0};
            left -= run;
            c16 = 0;
            ++rt;
            if (rt == P.L[l].n_rt) { rt = 0; ++l; }                       // (a task that ends here never looks at the layer again)
            return true;
        }
        const int run = min(left, P.n16 - c16), pieces = run <= P.max16 ? 1 : (run + P.max16 - 1) / P.max16;
        ps = Pass{0, rt, c16, pieces == 1 ? run : (run + pieces - 1) / pieces, s_lo, s_hi, path};
        if (SEQ) {                                                       // (such a task is one chunk: all its passes are the same but for the path)
            if (++path < P.paths) return true;
            path = 0;
        }
        left -= ps.n;
        c16 += ps.n;
        if (c16 == P.n16) { c16 = 0; ++rt; }
        return true;
    }
};

// Which of the acc_ready barriers says that all MMAs of a task's pass have retired, and the parity of that phase.  A wait by parity tells a phase
// from the one before it and from no other, so whoever waits for a barrier waits for every phase of it in turn.  In a stream task the warps
// for the epilogues do that with the two of the alternating passes; the expanders, which publish the last pass only and may be several
// passes ahead of the MMAs when they come to it (as many as the unit ring holds, and a group without units all of them), have a barrier of its own.
struct Ready {
    int bar;
    uint32_t parity;
};
__host__ __device__ __forceinline__ Ready ready_of(bool stream, int pass_i, bool last) {
    return !stream ? Ready{0, (uint32_t)pass_i & 1u} : last ? Ready{2, 0u} : Ready{pass_i & 1, (uint32_t)(pass_i >> 1) & 1u};
}

// Segments of a row tile of stream tasks: the tasks that touch its n_cs pairs, the first of which is pair `first` of n_pairs.  No task
// is empty.  (pairs < kMaxPairs and tasks <= kMaxTasks: 32 bits hold the products)
__host__ __device__ __forceinline__ int segment_arrivals(uint32_t first, uint32_t n_cs, uint32_t tasks, uint32_t n_pairs) {
    return (int)(((first + n_cs) * tasks - 1u) / n_pairs) - (int)(((first + 1u) * tasks - 1u) / n_pairs) + 1;
}

// K paths; DEQ: see above.  NL > 1: up to NL layers of at most 16 batch columns in one launch (stream tasks; each layer has
// its own x, of which the layers may share one).  SEQ (an instance with K = 1): path-major, for three paths.  Three accumulators
// leave room for 8 groups of columns at most, so wider batches expanded every tile two or three times; here a task
// is a pass per path on one accumulator, the sum of the scaled passes stays in tensor memory beside it, and up to 13 groups fit
// (5000 x 13824 at batch 200: each tile expanded once instead of three times).
template <int K, bool DEQ, int NL, bool SEQ>
__global__ void __launch_bounds__(threads_of(K, DEQ, SEQ, NL > 1), 1)
rabit_gemm_tc_kernel(const __grid_constant__ GemmParams<NL> P, const __grid_constant__ XMaps<NL> x_maps) {
    extern __shared__ unsigned char smem_raw[];
    // the swizzled x tiles need 1024-byte alignment; the launch reserves the slack
    unsigned char* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
    Control& S = *reinterpret_cast<Control*>(smem);
    const int tid = threadIdx.x, lane = tid & 31, warp = __shfl_sync(0xFFFFFFFFu, tid >> 5, 0);
    // The launch parameters sit in constant memory, cold in every launch (a first touch is a trip to L2, several in a row
    // between the dependency wait and the first MMA): touched here once, a 64-byte line per warp.  So is the tensor map.  (A
    // copy of them in shared memory is no better: the values are then not uniform to the compiler, and the issuers' loops
    // grow by 15 %.)
    if (warp < (int)((sizeof(GemmParams<NL>) + 63) / 64)) {
        const uint32_t word = reinterpret_cast<const uint32_t*>(&P)[warp * 16];
        asm volatile("" ::"r"(word));
    }
    if (warp == kFourthIssuer - 1 && lane < (NL == 1 ? 1 : P.n_layers)) asm volatile("prefetch.tensormap [%0];" ::"l"(&x_maps.map[NL == 1 ? 0 : lane]) : "memory");
    auto layer = [&](const Pass& ps) -> const GemmLayer& { return P.L[NL == 1 ? 0 : ps.l]; };
    unsigned char* ring = smem + kControlBytes;
    unsigned char* w_ring = ring + P.stages * P.stage_bytes;
    constexpr int n_ops = DEQ ? 1 : K;                            // operand units (and accumulators) per step
    constexpr int n_groups = n_ops == 3 || SEQ ? 3 : 4;                  // expander groups at work
    constexpr int max_acc = most_acc(K, DEQ, SEQ), n_fourth = max_acc > 3 ? 1 : 0;   // (n_fourth: whether there is a fourth issuing warp)
    const int stages = P.stages, w_stages = P.w_stages, units = P.units, x_steps = P.x_steps, n_acc = P.n_acc;
    const int stage_bytes = P.stage_bytes;
    volatile int* abort_flag = &S.abort_flag;
    // Split contraction: the CTAs of a cluster work on the same task, rank r taking the r-th part of the steps; their
    // partial results meet through distributed shared memory at the end (such a task is one pass).
    const int split = NL == 1 ? P.split : 1;
    uint32_t crank = 0;
    if (split > 1) asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(crank));
    const int task = split > 1 ? (int)blockIdx.x / split : (int)blockIdx.x;

    if (warp == 1) {                                              // (all of them, whatever the rings use: a lane each)
        if (lane < kMaxStages) { mbar_init(smem_u32(&S.full[lane]), 1); mbar_init(smem_u32(&S.empty[lane]), n_acc); }
        if (lane < kMaxWStages) { mbar_init(smem_u32(&S.w_full[lane]), 1); mbar_init(smem_u32(&S.w_empty[lane]), 4 * n_groups); }
        if (lane < kMaxUnits) { mbar_init(smem_u32(&S.a_ready[lane]), 4); mbar_init(smem_u32(&S.a_empty[lane]), 1); }
        if (lane == 0) {
            for (int i = 0; i < 3; ++i) mbar_init(smem_u32(&S.acc_ready[i]), n_acc);
            for (int i = 0; i < 2; ++i) mbar_init(smem_u32(&S.acc_empty[i]), NL > 1 ? 4 : kExpandWarps);
            S.abort_flag = 0;
            S.x_begun = -1;
#ifdef RABIT_CHECKED
            mbar_init(smem_u32(&S.never), 1);
#endif
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    if (split > 1) asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");   // (awaited before the exchange: every CTA of the cluster runs)
    const PassWalker<NL, SEQ> first_pass(P, task, (int)crank);
    // Output scales of the row whose accumulators this thread reads: loaded when a pass begins, converted (which waits for
    // them) when it ends.
    unsigned short graw[K];
    auto load_scales = [&](const Pass& ps) {
        if (!RABIT_IN_RANGE(ps.rt >= 0 && ps.rt < layer(ps).n_rt && ps.path >= 0 && ps.path < P.paths)) return;
#pragma unroll
        for (int k = 0; k < K; ++k)
            asm volatile("ld.global.nc.u16 %0, [%1];" : "=h"(graw[k]) : "l"(layer(ps).g + (size_t)(SEQ ? ps.path : k) * layer(ps).Mp + ps.rt * kTileM + (warp & 3) * 32 + lane));
    };
    auto scale = [&](int k) {
        unsigned short r;
        asm volatile("mov.b16 %0, %1;" : "=h"(r) : "h"(graw[k]));
        return __half2float(__ushort_as_half(r));
    };

    // SEQ: sum of the scaled passes before the last, 16 columns of group c
    [[maybe_unused]] auto path_sum = [&](int c, float (&v)[16]) {
        uint32_t d[16];
        tmem_ld16(__shfl_sync(0xFFFFFFFFu, S.tmem_base, 0) + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)((P.max16 + c) * kGroupCols), d);
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
        for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(d[i]);
    };

    // Stream: a pass's sums of this thread's row, batch columns [c0, c0 + n) (its scales are on their way).  A segment that is a whole row tile is stored;
    // otherwise every output goes into its 64-bit accumulate word with one integer atomic (as in rabit_gemv_f16.cu: fixed-point grid
    // of the packer, a segment of s slices shifted by s * 2^fix_bits, arrivals in bits 55..62, bit 63 = non-finite), and the thread
    // whose add completes a word rounds it to fp16, stores y and clears it.
    [[maybe_unused]] auto publish = [&](auto cols, auto is_last, const Pass& ps, int pass_i, int c0) {
        constexpr int n = decltype(cols)::value;
        constexpr bool last = decltype(is_last)::value;
        const GemmLayer& L = layer(ps);
        const int q = warp & 3, row = ps.rt * kTileM + q * 32 + lane, n_slices = (ps.s_hi - ps.s_lo + kSliceSteps - 1) / kSliceSteps, set = pass_i & 1;
        // (in registers: read from the parameters between the atomics, each would be a wait)
        const int M = L.M, Mp = L.Mp, n_cs = L.n_cs, fix_bits = L.fix_bits, n_here = P.batch - c0;
        const float inv_unit = L.inv_unit, unit = L.unit, limit = L.limit * (float)n_slices;
        __half* const y = L.y + (size_t)c0 * M + row;
        unsigned long long* const word = L.acc + (size_t)c0 * Mp + row;
        const int arrivals = segment_arrivals((uint32_t)(L.pair0 + ps.rt * n_cs), (uint32_t)n_cs, (uint32_t)P.n_tasks, (uint32_t)P.n_groups);
        const uint32_t from = __shfl_sync(0xFFFFFFFFu, S.tmem_base, 0) + ((uint32_t)(32 * q) << 16) + (uint32_t)(set * n_acc * kGroupCols + c0);
        const Ready ready = ready_of(true, pass_i, last);
        mbar_wait(smem_u32(&S.acc_ready[ready.bar]), ready.parity, abort_flag);
        __syncwarp();
        fence_after();
        float v[n];
#pragma unroll
        for (int i = 0; i < n; ++i) v[i] = 0.f;
#pragma unroll
        for (int m = 0; m < max_acc; ++m) {
            if (n_ops == 1 && m >= n_acc) break;
            uint32_t d[n];
            if constexpr (n == 16) tmem_ld16(from + (uint32_t)(m * kGroupCols), d);
            else tmem_ld4(from + (uint32_t)(m * kGroupCols), d);
            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
            const float gm = DEQ ? 1.f : scale(n_ops == 1 ? 0 : m);
#pragma unroll
            for (int i = 0; i < n; ++i) v[i] = fmaf(gm, __uint_as_float(d[i]), v[i]);
        }
        fence_before();
        __syncwarp();
        if (!last && lane == 0) mbar_arrive(smem_u32(&S.acc_empty[set]));     // (nothing follows the last pass)
        if (n_slices == n_cs) {
#pragma unroll
            for (int i = 0; i < n; ++i)
                if (i < n_here && row < M) y[(size_t)i * M] = __float2half_rn(v[i]);
            return;
        }
        // inf or NaN: finite inputs cannot get beyond the limit
        const unsigned long long bias = (unsigned long long)((long long)n_slices << fix_bits) + (1ULL << 55);
        auto bad = [&](int i) { return !(fabsf(v[i] * inv_unit) < limit); };
        auto contribution = [&](int i) { return (unsigned long long)(bad(i) ? 0LL : __float2ll_rn(v[i] * inv_unit)) + bias; };
        auto poison = [&](int i) {                               // sticky: the add that follows never carries into bit 63
            if (bad(i) && i < n_here && RABIT_IN_RANGE(row >= 0 && row < Mp && c0 + i < RABIT_LUT_MAX_BATCH)) atomicOr(word + (size_t)i * Mp, 1ULL << 63);
        };
        if constexpr (n == kGroupCols) {
            // (many in a row: no branch between the adds.  20000 x 1024 at 16 rows 9.25 -> 8.95 us; with four a thread 4096 x 4096 7.35 -> 7.45)
            uint32_t bads = 0u;
#pragma unroll
            for (int i = 0; i < n; ++i) bads |= bad(i) ? 1u : 0u;
            if (bads != 0u) [[unlikely]] {
#pragma unroll
                for (int i = 0; i < n; ++i) poison(i);
            }
        }
        unsigned long long old[n];
        // all atomics of the thread back to back: nothing between them that could wait for an answer
#pragma unroll
        for (int i = 0; i < n; ++i) {
            old[i] = 0ULL;
            if constexpr (n != kGroupCols) poison(i);
            if (i < n_here && RABIT_IN_RANGE(row >= 0 && row < Mp && c0 + i < RABIT_LUT_MAX_BATCH)) old[i] = atomicAdd(word + (size_t)i * Mp, contribution(i));
        }
#pragma unroll
        for (int i = 0; i < n; ++i) {
            if (i >= n_here || (int)((old[i] >> 55) & 0xFFu) != arrivals - 1) continue;       // other segments are still to come
            const unsigned long long sum = (old[i] & kSumMask) + (contribution(i) & kSumMask);
            const long long total = (long long)sum - ((long long)n_cs << fix_bits);
            const bool poisoned = bad(i) || (old[i] >> 63) != 0;
            if (row < M) y[(size_t)i * M] = poisoned ? __ushort_as_half((unsigned short)0x7FFF) : __float2half_rn(__ll2float_rn(total) * unit);
            word[(size_t)i * Mp] = 0ULL;                         // resting state for the next call
        }
    };

    auto weight_stages = [](const Pass& ps) { return (ps.s_hi - ps.s_lo + kWSteps - 1) / kWSteps; };
    // weight stage j of a pass into slot `slot` (these do not depend on the stream's past)
    auto load_weights = [&](const Pass& ps, int j, int slot) {
        const GemmLayer& L = layer(ps);
        const int rt = ps.rt, n_ct = L.n_ct, ct0 = 2 * (ps.s_lo + kWSteps * j), cts = min(kWTiles, min(2 * ps.s_hi, n_ct) - ct0);
        const uint32_t bar = smem_u32(&S.w_full[slot]), dst = smem_u32(w_ring + slot * (K * kWBytes));
        if (!RABIT_IN_RANGE(rt >= 0 && rt < L.n_rt && ps.path >= 0 && ps.path < P.paths && ct0 >= 0 && cts > 0 && ct0 + cts <= n_ct && L.N == n_ct * RABIT_TILE_COLS && slot < w_stages &&
                            dst + K * kWBytes <= smem_u32(smem_raw) + smem_bytes())) return;
        mbar_expect_tx(bar, (uint32_t)(K * cts * (RABIT_TILE_BYTES + RABIT_TILE_COLS * 2)));
#pragma unroll
        for (int k = 0; k < K; ++k) {
            bulk_g2s(dst + k * kWTiles * RABIT_TILE_BYTES, L.bits + ((SEQ ? (size_t)rt * P.paths + ps.path : (size_t)rt * K + k) * n_ct + ct0) * RABIT_TILE_BYTES, cts * RABIT_TILE_BYTES, bar);
            bulk_g2s(dst + K * kWTiles * RABIT_TILE_BYTES + k * kWTiles * RABIT_TILE_COLS * 2, L.h + (size_t)(SEQ ? ps.path : k) * L.N + (size_t)ct0 * RABIT_TILE_COLS,
                     cts * RABIT_TILE_COLS * 2, bar);
        }
    };
    // the weight stages of all passes in order; `next` starts one if its slot is free or becomes free
    struct WeightFeed {
        PassWalker<NL, SEQ> w;
        Pass ps;
        int j, issued;
        Walk at;
        bool more;
    };
    WeightFeed feed{first_pass, Pass{}, 0, 0, Walk{0}, false};
    auto feed_next = [&](bool elected) {                         // false: gave up (lane by lane: nothing below may wait for the other lanes)
        if (feed.issued >= w_stages && !mbar_wait(smem_u32(&S.w_empty[feed.at.slot]), feed.at.lap ^ 1u, abort_flag)) return false;
        if (elected) load_weights(feed.ps, feed.j, feed.at.slot);
        ++feed.issued;
        feed.at.step(1, w_stages);
        if (++feed.j == weight_stages(feed.ps)) { feed.j = 0; feed.more = feed.w.next(P, feed.ps); }
        return true;
    };
    if (warp == 0) {
        const bool elected = elect_one();
        feed.more = feed.w.next(P, feed.ps);
        while (feed.more && feed.issued < w_stages) feed_next(elected);
        __syncwarp();
    }
    asm volatile("griddepcontrol.wait;" ::: "memory");
    // Tensor memory is taken only after the dependency wait: a CTA that held some while the kernel before it in the stream
    // still had CTAs about to allocate would keep that kernel, and with it itself, waiting for good.
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(&S.tmem_base)) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    fence_before();
    __syncthreads();
    fence_after();
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const uint32_t tmem_base = __shfl_sync(0xFFFFFFFFu, S.tmem_base, 0);   // (one value per warp: the MMA operands then live in uniform registers)

    if (warp == 0) {
        // ===================================== producer =====================================
        const bool elected = elect_one();
        int it = 0, w_at = 0;                                    // x and weight stages begun, over all passes
        bool go = true;
        Walk at{0};
        PassWalker<NL, SEQ> w = first_pass;
        Pass ps;
        while (go && w.next(P, ps)) {
            const int boxes = (ps.n + P.box16 - 1) / P.box16;
            const uint32_t box_bytes = (uint32_t)(P.box16 * (kGroupCols * kStepCols * 2) * x_steps), tx = boxes * box_bytes;   // (what lies outside x arrives as zeros)
            for (int s = ps.s_lo; s < ps.s_hi; s += x_steps, ++it) {
                if ((s - ps.s_lo) % kWSteps == 0) {                 // (x_steps divides kWSteps)
                    ++w_at;                                      // two stages behind the ring's depth: never held up by the stage in use
                    while (go && feed.more && feed.issued < w_at + w_stages - 2) go = feed_next(elected);
                    if (!go) break;
                }
                const uint32_t bar = smem_u32(&S.full[at.slot]), dst = smem_u32(ring + at.slot * stage_bytes);
#ifdef RABIT_CHECKED
                if (it == P.withhold && !mbar_wait(smem_u32(&S.never), 0u, abort_flag)) { go = false; break; }
#endif
                if (it >= stages && !mbar_wait(smem_u32(&S.empty[at.slot]), at.lap ^ 1u, abort_flag)) { go = false; break; }
                if (elected && RABIT_IN_RANGE(at.slot < stages && tx <= (uint32_t)stage_bytes && dst + tx <= smem_u32(w_ring) && ps.c16 >= 0 && ps.c16 + ps.n <= P.n16)) {
                    mbar_expect_tx(bar, tx);
                    if (x_steps > 1) {
                        tma_load_3d(dst, &x_maps.map[NL == 1 ? 0 : ps.l], 0, ps.c16 * kGroupCols, s, bar);
                    } else {
                        for (int c = 0; c < boxes; ++c) tma_load_2d(dst + c * box_bytes, &x_maps.map[NL == 1 ? 0 : ps.l], s * kStepCols, (ps.c16 + c * P.box16) * kGroupCols, bar);
                    }
                }
                at.step(1, stages);
            }
        }
        if (elected) {
            S.w_begun = feed.issued;
            *(volatile int*)&S.x_begun = it;
        }
        __syncwarp();
    } else if (warp < 4 || (n_fourth && warp == kFourthIssuer)) {
        // ===================================== MMA issuers =====================================
        // Warp 1 + m issues the units u = m, m + n_acc, ... into accumulator m.  (The whole warp walks the loop, one elected lane
        // issues: see the header.)
        auto issue_units = [&](auto acc) {
            constexpr int m = decltype(acc)::value;
            const bool elected = elect_one();
            int pass_i = 0;
            Walk uw{m}, xw{0};                                   // units of this accumulator, x stages
            const int u_stride = n_ops == 1 ? n_acc : 1;         // steps from one of its units to the next
            const uint32_t full0 = smem_u32(&S.full[0]), empty0 = smem_u32(&S.empty[0]), a_ready0 = smem_u32(&S.a_ready[0]), a_empty0 = smem_u32(&S.a_empty[0]);
            const uint64_t bdesc0 = umma_desc(smem_u32(ring));
            const uint32_t a0 = tmem_base + (uint32_t)P.a_col, d0 = tmem_base + (uint32_t)(m * P.max16 * kGroupCols);
            const uint32_t step_bytes = (uint32_t)stage_bytes / (uint32_t)x_steps;
            int steps_before = 0;                                // of earlier passes
            PassWalker<NL, SEQ> w = first_pass;
            Pass ps;
            while (w.next(P, ps)) {
                const uint32_t idesc = __shfl_sync(0xFFFFFFFFu, umma_idesc(ps.n * kGroupCols), 0);
                // the epilogue of the pass that had these accumulators has read them
                const int set = NL > 1 ? pass_i & 1 : 0;
                const uint32_t d = NL > 1 ? __shfl_sync(0xFFFFFFFFu, d0 + (uint32_t)(set * n_acc * kGroupCols), 0) : d0;
                if (NL > 1 ? pass_i > 1 : pass_i > 0) mbar_wait(smem_u32(&S.acc_empty[set]), (NL > 1 ? (pass_i >> 1) - 1 : pass_i - 1) & 1, abort_flag);
                ++pass_i;
                if (!RABIT_IN_RANGE(ps.n >= 1 && ps.n <= P.max16 && (m + 1) * P.max16 * kGroupCols <= P.a_col && P.a_col + units * kUnitCols <= 512)) break;
                uint32_t accumulate = 0u;
                const int s_lo = __shfl_sync(0xFFFFFFFFu, ps.s_lo, 0), s_hi = __shfl_sync(0xFFFFFFFFu, ps.s_hi, 0);
                const int n_ct = NL == 1 ? P.L[0].n_ct : __shfl_sync(0xFFFFFFFFu, P.L[ps.l].n_ct, 0);
                for (int s = s_lo; s < s_hi; s += x_steps) {
                    const int n_here = min(x_steps, s_hi - s);
                    mbar_wait_stage(full0 + xw.slot * 8, xw.lap, abort_flag, &S.x_begun);
                    const uint64_t bdesc = bdesc0 + (uint64_t)((xw.slot * stage_bytes) >> 4);
                    int si = n_ops == 1 ? (m - (steps_before + s - s_lo)) & (n_acc - 1) : 0;   // (1, 2 or 4 accumulators)
                    auto issue = [&](uint32_t a, int step, bool first) {
                        const uint64_t bd = bdesc + (uint64_t)((step * step_bytes) >> 4);
                        umma_f16_ts(d, a, bd, idesc, first ? accumulate : 1u);
                        umma_f16_ts(d, a + 8, bd + 2, idesc, 1u);
                        if (2 * (s + step) + 1 < n_ct) {         // (the last step may hold one column tile)
                            umma_f16_ts(d, a + 16, bd + 4, idesc, 1u);
                            umma_f16_ts(d, a + 24, bd + 6, idesc, 1u);
                        }
                    };
                    // with two paths two units at a time: their waits overlap (one at a time the two issuers were what layers with
                    // few batch columns waited for; with one or three paths this measured slower)
                    for (; n_ops == 2 && si + u_stride < n_here; si += 2 * u_stride) {
                        Walk second = uw;
                        second.step(n_acc, units);
                        const bool r1 = mbar_try_wait(a_ready0 + uw.slot * 8, uw.lap), r2 = mbar_try_wait(a_ready0 + second.slot * 8, second.lap);
                        if (!r1) mbar_wait(a_ready0 + uw.slot * 8, uw.lap, abort_flag);
                        if (!r2) mbar_wait(a_ready0 + second.slot * 8, second.lap, abort_flag);
                        fence_after();
                        if (elected) {
                            issue(a0 + uw.slot * kUnitCols, si, true);
                            umma_commit(a_empty0 + uw.slot * 8);
                            issue(a0 + second.slot * kUnitCols, si + u_stride, false);
                            umma_commit(a_empty0 + second.slot * 8);
                        }
                        accumulate = 1u;
                        __syncwarp();
                        uw = second;
                        uw.step(n_acc, units);
                    }
                    for (; si < n_here; si += u_stride) {
                        mbar_wait(a_ready0 + uw.slot * 8, uw.lap, abort_flag);
                        fence_after();
                        if (elected) {
                            issue(a0 + uw.slot * kUnitCols, si, true);
                            umma_commit(a_empty0 + uw.slot * 8);
                        }
                        accumulate = 1u;
                        __syncwarp();
                        uw.step(n_acc, units);
                    }
                    if (elected) umma_commit(empty0 + xw.slot * 8);
                    __syncwarp();
                    xw.step(1, stages);
                }
                steps_before += s_hi - s_lo;
                const uint32_t passed = __shfl_sync(0xFFFFFFFFu, smem_u32(&S.acc_ready[ready_of(NL > 1, pass_i - 1, w.left <= 0).bar]), 0);
                if (elected) umma_commit(passed);
                __syncwarp();
            }
        };
        if (warp == 1) issue_units(std::integral_constant<int, 0>{});
        else if (warp == 2 && n_acc > 1) issue_units(std::integral_constant<int, 1>{});
        else if (warp == 3 && n_acc > 2) issue_units(std::integral_constant<int, 2>{});
        else if (n_fourth && warp == kFourthIssuer && n_acc > 3) issue_units(std::integral_constant<int, 3>{});
    } else if (warp < kFourthIssuer) {
        // ============================ expanders, then epilogue ============================
        const int grp = (warp - 4) >> 2, q = warp & 3;        // tensor-memory lanes this warp may touch: 32q .. 32q + 31
        const int gq = lane >> 2, tq = lane & 3;
        const uint32_t lane_base = tmem_base + ((uint32_t)(32 * q) << 16);
        // bits 2q and 2q + 1 of a byte to its top two: a multiplication by a power of two, 64 >> 2q, that the compiler does not know to be one (it
        // goes to the multiply-add pipe instead of the one that the byte permutes and logic instructions fill)
        const uint32_t keep = 0x03030303u << (2 * q);
        uint32_t up = 64u >> (2 * q);
        asm volatile("" : "+r"(up));
        // Integer instructions take two issue clocks each and bound this loop (80 of them a unit and warp are the expansion
        // itself), so everything around them is kept in few registers that only step: a group always has the same path, and
        // its units alternate between the same one or two places in tensor memory.
        const int path = grp % n_ops;
        constexpr int kStepsOn = n_groups / n_ops;            // steps from one of the group's units to its next
        const uint32_t dst0 = lane_base + (uint32_t)(P.a_col + grp * kUnitCols), dst_sum = 2 * dst0 + (units > n_groups ? n_groups * kUnitCols : 0);
        const uint32_t bar0 = smem_u32(&S.a_empty[grp]), bar_sum = 2 * bar0 + (units > n_groups ? n_groups * 8u : 0u);
        constexpr uint32_t kBack = (uint32_t)(offsetof(Control, a_empty) - offsetof(Control, a_ready));   // from a unit's a_empty barrier to its a_ready
        const int lap_bit = units > n_groups ? 1 : 0;
        const uint32_t w_full0 = smem_u32(&S.w_full[0]), w_empty0 = smem_u32(&S.w_empty[0]);
        const uint32_t bits0 = smem_u32(w_ring) + lane * 16 + (DEQ ? 0 : path * kWTiles * RABIT_TILE_BYTES);
        const uint32_t h0 = smem_u32(w_ring) + K * kWTiles * RABIT_TILE_BYTES + 8 * tq + (DEQ ? 0 : path * kWTiles * RABIT_TILE_COLS * 2);
        uint32_t dst = dst0, bar = bar0, done = 0;            // done: the group's units so far
        Walk ww{0};
        int pass_i = 0, u0 = 0;
        PassWalker<NL, SEQ> w = first_pass;
        Pass ps;
        while (w.next(P, ps)) {
            const GemmLayer& L = layer(ps);
            const int n_ct = L.n_ct;
            __half2 g_rows[DEQ ? K : 1][2][2];                 // DEQ: output scales of this thread's rows (row block, row half), both halves alike
            if (DEQ) {
#pragma unroll
                for (int k = 0; k < K; ++k)
#pragma unroll
                    for (int pi = 0; pi < 2; ++pi)
#pragma unroll
                        for (int rh = 0; rh < 2; ++rh)
                            g_rows[k][pi][rh] = __half2half2(L.g[(size_t)k * L.Mp + ps.rt * kTileM + 32 * q + 16 * pi + gq + 8 * rh]);
            }
            if (NL == 1 || w.left <= 0) load_scales(ps);
            int first = ((grp - u0 % n_groups + n_groups) % n_groups) / n_ops;   // the group's first step of the pass, and (unless its stride does not divide them) of each weight stage
            for (int j = 0; j < weight_stages(ps) && grp < n_groups; ++j) {
                const int step0 = ps.s_lo + j * kWSteps, n_here = min(kWSteps, ps.s_hi - step0), whole = min(n_here, n_ct / 2 - step0);   // steps with two column tiles
                uint32_t bits = bits0 + ww.slot * (K * kWBytes) + first * (2 * RABIT_TILE_BYTES), hs = h0 + ww.slot * (K * kWBytes) + first * (kStepCols * 2);
                mbar_wait_stage(w_full0 + ww.slot * 8, ww.lap, abort_flag, &S.x_begun);
                int sj = first;
                for (; sj < n_here; sj += kStepsOn) {
                    const uint32_t parity = ((done >> lap_bit) & 1u) ^ 1u;                  // (the first time round this is the barrier's previous phase: free)
                    const bool both = sj < whole;
                    if (!RABIT_IN_RANGE((dst & 0xFFFFu) - (tmem_base & 0xFFFFu) >= (uint32_t)P.a_col && (dst & 0xFFFFu) - (tmem_base & 0xFFFFu) + kUnitCols <= 512u && sj < kWSteps && ww.slot < w_stages &&
                                        bar >= smem_u32(&S.a_empty[0]) && bar <= smem_u32(&S.a_empty[units - 1]))) break;
                    auto load = [&](int kk, int ct2) {
                        TileIn t;
                        t.w = lds_v4(bits + (kk * kWTiles + ct2) * RABIT_TILE_BYTES);
#pragma unroll
                        for (int ah = 0; ah < 2; ++ah) t.h[ah] = lds_v2(hs + (kk * kWTiles * RABIT_TILE_COLS + 32 * ct2 + 16 * ah) * 2);
                        return t;
                    };
                    // a tile of path kk into operand registers o[row block][16-column half, row half, column pair]
                    auto expand = [&](const TileIn& t, int kk, uint32_t (&o)[2][8]) {
                        // (dequantised, three paths: the multiply-add pipe has enough to do already, 14336 x 4096 at 16 rows 21.2 -> 20.9 us; wider passes 6 % slower)
                        auto top = [&](uint32_t w) { return DEQ && K == 3 && NL > 1 ? (w & keep) << (6 - 2 * q) : mul_lo(w & keep, up); };
                        const uint32_t word[4] = {top(t.w.x), top(t.w.y), top(t.w.z), top(t.w.w)};
#pragma unroll
                        for (int ah = 0; ah < 2; ++ah)
#pragma unroll
                            for (int rh = 0; rh < 2; ++rh)
#pragma unroll
                                for (int pair = 0; pair < 2; ++pair) {
                                    // bytes [0, c0, 0, c1]: row block 2q + 1's bits at 15 and 31, row block 2q's one below, nothing else
                                    const uint32_t v = __byte_perm(word[2 * ah + rh], 0u, pair ? 0x3424 : 0x1404);
                                    const uint32_t hp = pair ? t.h[ah].y : t.h[ah].x, odd = (v & 0x80008000u) ^ hp;
                                    // As an fp16 number v is 0 or 2 (the bit at 14) with the sign that odd has beside h, so h - v * odd is h or h - 2 h (exact; NaN if h is infinite)
                                    const __half2 even2 = __hfma2(*reinterpret_cast<const __half2*>(&v), __hneg2(*reinterpret_cast<const __half2*>(&odd)), *reinterpret_cast<const __half2*>(&hp));
#pragma unroll
                                    for (int pi = 0; pi < 2; ++pi) {
                                        const __half2 m = pi ? *reinterpret_cast<const __half2*>(&odd) : even2;
                                        uint32_t& a = o[pi][4 * ah + 2 * rh + pair];
                                        const __half2 r = DEQ ? __hfma2(g_rows[DEQ ? kk : 0][pi][rh], m, *reinterpret_cast<const __half2*>(&a)) : m;
                                        a = *reinterpret_cast<const uint32_t*>(&r);
                                    }
                                }
                    };
                    auto store = [&](int ct2, const uint32_t (&o)[2][8]) {
                        tmem_st_16x256b_x2(dst + ct2 * 16, o[0]);
                        tmem_st_16x256b_x2(dst + ct2 * 16 + (16u << 16), o[1]);
                    };
                    uint32_t o[2][8];
                    if constexpr (DEQ) {
                        mbar_wait(bar, parity, abort_flag);
                        fence_after();
                        // dequantised: sum_k +-g_k[row] h_k[col], accumulated from the last (smallest) path to the first with one fused
                        // multiply-add per path
                        for (int ct2 = 0; ct2 < (both ? 2 : 1); ++ct2) {
#pragma unroll
                            for (int i = 0; i < 8; ++i) o[0][i] = o[1][i] = 0u;
#pragma unroll
                            for (int kk = K - 1; kk >= 0; --kk) expand(load(kk, ct2), kk, o);
                            store(ct2, o);
                        }
                    } else if constexpr (K == 3) {
                        // Three groups have fewer warps to hide a unit's steps behind: its words are on their way and its place is asked for
                        // first (5000 x 13824 at 16 / 48 rows 23.2 / 26.8 -> 22.0 / 25.2 us; with four groups no gain, with one path 2 % slower).
                        const TileIn t0 = load(0, 0);
                        const bool empty = mbar_test_wait(bar, parity);
                        TileIn t1;
                        if (both) t1 = load(0, 1);
                        expand(t0, 0, o);
                        if (!empty) mbar_wait(bar, parity, abort_flag);
                        fence_after();
                        store(0, o);
                        if (both) { expand(t1, 0, o); store(1, o); }
                    } else {
                        mbar_wait(bar, parity, abort_flag);
                        fence_after();
                        expand(load(0, 0), 0, o);
                        store(0, o);
                        if (both) { expand(load(0, 1), 0, o); store(1, o); }
                    }
                    bits += kStepsOn * 2 * RABIT_TILE_BYTES;
                    hs += kStepsOn * kStepCols * 2;
                    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
                    fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(bar - kBack);
                    dst = dst_sum - dst;
                    bar = bar_sum - bar;
                    ++done;
                }
                if (kWSteps % kStepsOn != 0) first = sj - n_here;
                __syncwarp();
                if (lane == 0) mbar_arrive(w_empty0 + ww.slot * 8);
                ww.step(1, w_stages);
            }
            u0 += (ps.s_hi - ps.s_lo) * n_ops;
            if (split > 1 && (!SEQ || ps.path == P.paths - 1)) break;   // the cluster's epilogue follows the role branches
            if constexpr (NL > 1) {
                // A pass that another one follows is published by warps of their own, while this one is expanded (its accumulators are not
                // those of the next); the last one by these, which are four times as many.
                if (w.left <= 0) publish(std::integral_constant<int, 4>{}, std::true_type{}, ps, pass_i, 4 * grp);
                ++pass_i;
                continue;
            }
            // ---- epilogue of this pass
            const Ready ready = ready_of(false, pass_i, false);
            mbar_wait(smem_u32(&S.acc_ready[ready.bar]), ready.parity, abort_flag);
            ++pass_i;
            fence_after();
            const int row = ps.rt * kTileM + q * 32 + lane;
            if constexpr (SEQ) {
                if (ps.path < P.paths - 1) {
                    // a path that is not the last: its scaled result joins the sum beside the accumulator
#pragma unroll 1
                    for (int c = grp; c < ps.n; c += kExpandGroups) {
                        const uint32_t acc = lane_base + (uint32_t)(c * kGroupCols), sum = acc + (uint32_t)(P.max16 * kGroupCols);
                        uint32_t d[16], t[16];
                        tmem_ld16(acc, d);
                        if (ps.path > 0) tmem_ld16(sum, t);
                        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                        const float g = scale(0);
#pragma unroll
                        for (int i = 0; i < 16; ++i) t[i] = __float_as_uint(fmaf(g, __uint_as_float(d[i]), ps.path > 0 ? __uint_as_float(t[i]) : 0.f));
                        tmem_st16(sum, t);
                    }
                    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
                    fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(smem_u32(&S.acc_empty[0]));
                    continue;
                }
            }
            if constexpr (NL == 1) {
#pragma unroll 1
                for (int c = grp; c < ps.n; c += kExpandGroups) {
                    float v[16];
#pragma unroll
                    for (int i = 0; i < 16; ++i) v[i] = 0.f;
                    if constexpr (SEQ) path_sum(c, v);
#pragma unroll
                    for (int m = 0; m < max_acc; ++m) {
                        if (n_ops == 1 && m >= n_acc) break;
                        uint32_t d[16];
                        tmem_ld16(lane_base + (uint32_t)((m * P.max16 + c) * kGroupCols), d);
                        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                        const float gm = DEQ ? 1.f : scale(n_ops == 1 ? 0 : m);
#pragma unroll
                        for (int i = 0; i < 16; ++i) v[i] = fmaf(gm, __uint_as_float(d[i]), v[i]);
                    }
                    const int b0 = (ps.c16 + c) * kGroupCols;
                    __half* yp = L.y + (size_t)b0 * L.M + row;
                    if (row < L.M) {
#pragma unroll
                        for (int i = 0; i < 16; ++i)
                            if (b0 + i < P.batch) yp[(size_t)i * L.M] = __float2half_rn(v[i]);
                    }
                }
            }
            fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&S.acc_empty[0]));
        }
    } else {
        // ============================ epilogues of a stream task's passes, but for the last ============================
        int pass_i = 0;
        PassWalker<NL, SEQ> w = first_pass;
        Pass ps;
        while (w.next(P, ps) && w.left > 0) {
            load_scales(ps);
            publish(std::integral_constant<int, kGroupCols>{}, std::false_type{}, ps, pass_i, 0);
            ++pass_i;
        }
    }

    if (split > 1) {
        // ---- epilogue of a split task.  Every CTA of the cluster holds a partial result in tensor memory.  Group c of 16
        //      batch columns is finished by CTA c % split: all CTAs send it that group's columns (already scaled by g_k and
        //      summed over the paths) into its receive buffer recv[its c / split][source rank][column][row], behind the rings.
        //      After the cluster barrier each CTA adds what it received in rank order and stores fp16.
        PassWalker<NL, SEQ> w = first_pass;
        Pass ps;
        w.next(P, ps);
        if (warp >= 4 && warp < kFourthIssuer) {
            mbar_wait(smem_u32(&S.acc_ready[0]), SEQ ? (P.paths - 1) & 1 : 0, abort_flag);
            fence_after();
        }
        __syncwarp();
        asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
        if (SEQ) cluster_sync_all();                           // the receive buffer lies in the rings: every CTA's are done with
        float* recv = reinterpret_cast<float*>(smem + P.recv_off);
        if (warp >= 4 && warp < kFourthIssuer) {
            const int grp = (warp - 4) >> 2, q = warp & 3, r_in = q * 32 + lane;
#pragma unroll 1
            for (int c = grp; c < ps.n; c += kExpandGroups) {
                float v[16];
#pragma unroll
                for (int i = 0; i < 16; ++i) v[i] = 0.f;
                if constexpr (SEQ) path_sum(c, v);
#pragma unroll
                for (int m = 0; m < max_acc; ++m) {
                    if (n_ops == 1 && m >= n_acc) break;
                    uint32_t d[16];
                    tmem_ld16(tmem_base + ((uint32_t)(32 * q) << 16) + (uint32_t)((m * P.max16 + c) * kGroupCols), d);
                    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                    const float gm = DEQ ? 1.f : scale(n_ops == 1 ? 0 : m);
#pragma unroll
                    for (int i = 0; i < 16; ++i) v[i] = fmaf(gm, __uint_as_float(d[i]), v[i]);
                }
                if (!RABIT_IN_RANGE((const unsigned char*)(recv + ((size_t)((c / split) * split + split) * kGroupCols) * kTileM) <= smem_raw + smem_bytes())) continue;
                const uint32_t dst = cluster_map(smem_u32(recv + ((size_t)((c / split) * split + crank) * kGroupCols) * kTileM + r_in), (uint32_t)(c % split));
#pragma unroll
                for (int i = 0; i < 16; ++i) st_cluster_f32(dst + (uint32_t)(i * kTileM * 4), v[i]);
            }
            fence_before();
        }
        __syncwarp();
        cluster_sync_all();
        if (warp >= 4 && warp < kFourthIssuer) {
            const int et = (warp - 4) * 32 + lane, r_in = et & (kTileM - 1), hh = et >> 7;  // four threads per row, every fourth column each
            const int row = ps.rt * kTileM + r_in;
            for (int c = (int)crank; c < ps.n; c += split)
#pragma unroll
                for (int i = hh; i < kGroupCols; i += kExpandGroups) {
                    const float* src = recv + ((size_t)((c / split) * split) * kGroupCols + i) * kTileM + r_in;
                    float sum = 0.f;
                    for (int r = 0; r < split; ++r) sum += src[(size_t)r * kGroupCols * kTileM];
                    const int b = (ps.c16 + c) * kGroupCols + i;
                    if (b < P.batch && row < P.L[0].M) P.L[0].y[(size_t)b * P.L[0].M + row] = __float2half_rn(sum);
                }
        }
    }

    // ---- teardown: everyone meets, then the allocating warp frees the tensor memory
    fence_before();
    __syncthreads();
    fence_after();
    auto free_tensor_memory = [&] { asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem_base) : "memory"); };
    const bool gave_up = *abort_flag != 0;                     // (the same for every thread: nobody sets it any more)
    if (warp == 1 && !gave_up) free_tensor_memory();
    if (gave_up) [[unlikely]] {
        // Copies and MMAs under way must not outlive the shared and tensor memory they work on.  (All of it in one branch of its
        // own: with the ordinary path running through it a launch took 0.1 us longer.)
        if (tid < kMaxAcc) mbar_init(smem_u32(&S.drained[tid]), 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        __syncthreads();
        const long long t0 = clock64();
        if ((warp >= 1 && warp <= 3) || (n_fourth && warp == kFourthIssuer)) {   // (an arrival once all that this lane issued has retired)
            const uint32_t bar = smem_u32(&S.drained[warp <= 3 ? warp - 1 : 3]);
            if (elect_one()) umma_commit(bar);
            __syncwarp();
            while (!mbar_try_wait(bar, 0u) && clock64() - t0 <= kWaitLimitCycles) { }
        } else if (tid == 0) {
            drain_ring(S.full, stages, S.x_begun, t0);
            drain_ring(S.w_full, w_stages, S.w_begun, t0);
        }
        fence_before();
        __syncthreads();
        fence_after();
        if (warp == 1) free_tensor_memory();
        if (tid == 0)
            for (int l = 0; l < (NL == 1 ? 1 : P.n_layers); ++l) atomicExch(P.L[l].status, 1u);
    }
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                                  const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_tiled_fn() {
    static const EncodeTiledFn fn = [] {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) == cudaSuccess && q == cudaDriverEntryPointSuccess)
            return (EncodeTiledFn)p;
        return (EncodeTiledFn) nullptr;
    }();
    return fn;
}

// Descriptor of x [batch][N] in boxes of 16 * box16 rows x 64 columns, or x_steps such boxes side by side.  A pure function of its arguments; the last few are
// remembered per thread (encoding one costs about a microsecond of host time).
cudaError_t x_tensor_map(const void* x, int N, int batch, int box16, int x_steps, CUtensorMap* out) {
    struct Entry { const void* x; int N, batch, box16, x_steps; CUtensorMap map; };
    static thread_local Entry recent[8];
    static thread_local int next = 0;
    for (const Entry& e : recent)
        if (e.x == x && e.N == N && e.batch == batch && e.box16 == box16 && e.x_steps == x_steps) { *out = e.map; return cudaSuccess; }
    EncodeTiledFn encode = encode_tiled_fn();
    if (!encode) return cudaErrorNotSupported;
    // (with several steps per box N is a multiple of 64, so that no box reads beyond a row)
    const cuuint64_t dims[3] = {(cuuint64_t)(x_steps > 1 ? kStepCols : N), (cuuint64_t)batch, (cuuint64_t)(N / kStepCols)};
    const cuuint64_t strides[2] = {(cuuint64_t)N * 2, (cuuint64_t)kStepCols * 2};
    const cuuint32_t box[3] = {(cuuint32_t)kStepCols, (cuuint32_t)(box16 * kGroupCols), (cuuint32_t)x_steps};
    const cuuint32_t estr[3] = {1, 1, 1};
    if (encode(out, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, x_steps > 1 ? 3 : 2, const_cast<void*>(x), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
               CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
        return cudaErrorInvalidValue;
    recent[next] = Entry{x, N, batch, box16, x_steps, *out};
    next = (next + 1) & 7;
    return cudaSuccess;
}

// ---- choosing the work split -------------------------------------------------------------------------

struct Plan {
    int chunks, chunk16, split, max16, tasks;        // chunks == 0: contiguous group ranges
    int stream;                                      // contiguous ranges of (row tile, slice) pairs
    int seq;                                         // path-major
    int stages, stage_bytes, x_steps, w_stages, box16, units, n_acc, recv_off;
    size_t smem;
    double clocks;                                   // estimate
};

// Ring, tensor-memory and shared-memory figures of passes of up to max16 groups; false if they do not fit.  The units are a
// multiple of the expander groups and of the accumulators (see Walk).
bool fill_resources(Plan& p, int K, bool deq, int steps, bool one_box) {
    const int n_ops = deq || p.seq ? 1 : K;
    const int recv_bytes = p.split > 1 ? (p.chunk16 + p.split - 1) / p.split * p.split * kGroupCols * kTileM * 4 : 0;
    if (p.max16 * kGroupCols > 256) return false;
    const int turn = n_ops == 3 || p.seq ? 3 : 4;
    auto free_units = [&](int n_acc) { return (512 - ((p.stream ? 2 : 1) * n_acc + p.seq) * p.max16 * kGroupCols) / kUnitCols; };   // (a stream: two sets of accumulators)
    // One operand per step: up to four accumulators, if every pass has a step for each (a stream's shortest one is the last slice) and x comes in
    // several steps a stage (every issuing warp sees every stage: with one step in each 3894 x 14304 at 42 18.6 -> 19.5 us) and
    // the contraction is long enough to pay for adding them up (8 steps, 2000 x 4096 at 64 7.1 -> 7.3; 16, 4096 x 4096 at 32 7.17 -> 7.26; 32,
    // 600 x 16384 at 20 8.35 -> 7.8).  One or two
    // issuing warps were what such layers waited for up to 64 batch columns (one path, 28672 x 8192 at 16 26.5 -> 25.5 us, 14336 x 4096 at 48 10.85 -> 10.45;
    // with two paths, whose two warps issue pairs of units, four of them are 2 to 4 % slower).
    p.n_acc = n_ops;
    if (n_ops == 1 && !p.seq)
        for (int more = 2; more <= std::min(most_acc(K, deq, false), one_box && (p.stream || steps >= 24) ? kMaxAcc : 2) && steps >= more && free_units(more) >= (more == 2 ? turn : 2 * turn); more *= 2) p.n_acc = more;
    if (free_units(p.n_acc) < turn) return false;
    p.units = free_units(p.n_acc) >= 2 * turn ? 2 * turn : turn;
    const int step_bytes = (p.max16 + p.box16 - 1) / p.box16 * p.box16 * kGroupCols * kStepCols * 2;
    const int room = (226 - 1) * 1024 - kControlBytes - (p.seq ? 0 : recv_bytes);
    // as many steps per x stage (one copy of the producer, which needs some 600 clocks for each) as leave three stages
    for (p.x_steps = one_box ? 4 : 1;; p.x_steps /= 2) {
        p.stage_bytes = step_bytes * p.x_steps;
        p.stages = std::max(0, std::min(kMaxStages, (room - 3 * K * kWBytes) / p.stage_bytes));
        if (p.stages >= (p.x_steps > 1 ? 3 : 4)) break;
        if (p.x_steps == 1) return false;
    }
    p.w_stages = std::min(kMaxWStages, (room - p.stages * p.stage_bytes) / (K * kWBytes));
    // Never so little that two CTAs could share an SM: each takes all of its tensor memory, and of two clusters waiting
    // crosswise for each other's neither would ever get it.
    p.recv_off = kControlBytes + p.stages * p.stage_bytes + p.w_stages * K * kWBytes;
    size_t used = (size_t)p.recv_off;
    if (p.seq) {                                             // the receive buffer takes the rings' place
        p.recv_off = kControlBytes;
        used = std::max<size_t>(used, kControlBytes + recv_bytes);
    } else {
        used += recv_bytes;
    }
    p.smem = std::max<size_t>(1024 + used, 152 * 1024);
    return p.smem <= 226 * 1024;
}

// Clocks of a (step, path) unit, fitted on B200: four MMAs of the pass's batch columns, or the expansion of its two sign tiles
// (its share of issue slots and the hand-overs around it; more if a group has only one unit's room in tensor memory and has
// to wait for its MMAs).  Path-major: one warp issues everything and is the bound up to 16 groups (390 clocks at 7 groups, 510 at 13),
// so that it pays only where the others expand a tile several times: 5000 x 13824 at batch 130 / 200 71 -> 56 / 75 -> 68 us.
double unit_clocks(int n16, const Plan& p, int n_ops) {
    if (p.seq) return 250.0 + 20.0 * n16;
    return std::max(32.0 * n16 + 52.0, p.units >= 2 * (n_ops == 3 ? 3 : 4) ? 180.0 + 8.0 * n16 : n_ops == 3 ? 345.0 : 300.0);
}

// (stream: the form for contiguous ranges of up to kMaxGroup layers)
template <int NL>
const void* kernel_of(int K, bool deq) {
    if (K == 1) return deq ? (const void*)rabit_gemm_tc_kernel<1, true, NL, false> : (const void*)rabit_gemm_tc_kernel<1, false, NL, false>;
    if (K == 2) return deq ? (const void*)rabit_gemm_tc_kernel<2, true, NL, false> : (const void*)rabit_gemm_tc_kernel<2, false, NL, false>;
    return deq ? (const void*)rabit_gemm_tc_kernel<3, true, NL, false> : (const void*)rabit_gemm_tc_kernel<3, false, NL, false>;
}
const void* kernel_for(int K, bool deq, bool stream = false, bool seq = false) {
    return seq ? (const void*)rabit_gemm_tc_kernel<1, false, 1, true> : stream ? kernel_of<kMaxGroup>(K, deq) : kernel_of<1>(K, deq);
}

// Function attributes are per device.
cudaError_t prepare_kernel(int K, bool deq, int device, bool stream = false, bool seq = false) {
    static bool done[64][13] = {};
    const int slot = device >= 0 && device < 64 ? device : 0, inst = seq ? 12 : 4 * (K - 1) + (stream ? 2 : 0) + (deq ? 1 : 0);
    if (done[slot][inst] && slot == device) return cudaSuccess;
    cudaError_t e = cudaFuncSetAttribute(kernel_for(K, deq, stream, seq), cudaFuncAttributeMaxDynamicSharedMemorySize, 226 * 1024);
    if (e == cudaSuccess) done[slot][inst] = true;
    return e;
}

// How many clusters of `split` CTAs of this kernel the device places at once (a cluster sits inside one GPC).
int resident_clusters(const void* kernel, int threads, int split, size_t smem, int sms) {
    cudaLaunchConfig_t q = {};
    q.gridDim = dim3((unsigned int)((sms / split) * split));
    q.blockDim = dim3((unsigned int)threads);
    q.dynamicSmemBytes = smem;
    cudaLaunchAttribute qa[1];
    qa[0].id = cudaLaunchAttributeClusterDimension;
    qa[0].val.clusterDim.x = (unsigned int)split;
    qa[0].val.clusterDim.y = 1;
    qa[0].val.clusterDim.z = 1;
    q.attrs = qa;
    q.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, kernel, &q) != cudaSuccess) { cudaGetLastError(); n = 0; }
    return n;
}

constexpr double kPassClocks = 3000.0;               // pipeline fill and epilogue of a pass that nothing overlaps
constexpr double kLaunchClocks = 8000.0;             // launch, first loads, last epilogue
constexpr double kExchangeClocks = 2500.0;           // exchange of a split task
// Streams, fitted to 470 shapes (128 to 28672 rows, 64 to 13824 columns, one to three paths, 9 and 16 batch rows) x their task counts (B200): launch, unit of
// one, two or three paths, a further pass in a range; and where a range ends in a part of a row tile, publishing that part (the atomics and their
// answers; those of earlier parts run beside the next pass) and the throughput of all such ends, in sums per clock over the GPU.  The split that
// they pick is 0.2 % slower than the best on average, 4.5 % at most.  (Every part counted, publishing at 800 clocks, a pass at 1300: 1.0 % and 17 %;
// 256 x 512 with two paths, whose two slices are better not split, 3.75 against 4.35 us, 14336 x 4096 with three paths 20.0 on 112 tasks against 18.55 on 148.)
// The dequantised form's one unit a step takes kStreamDeq more for every path after the first (4096 x 4096 and 14336 x 4096 at 16 rows with one, two and three paths).
constexpr double kStreamLaunch = 5600.0, kStreamUnit[3] = {195.0, 185.0, 175.0}, kStreamDeq = 210.0, kStreamPass = 1150.0, kStreamPublish = 2050.0, kStreamRate = 140.0;

// Task counts worth an estimate: equal parts of every row tile (or nearly), and one task per SM.  Never more tasks than pairs: an
// empty one would count among the arrivals of a row tile that it does not contribute to.  (Layers of unlike widths: parts for the
// widest are more than the narrow ones have pairs.)
template <typename F>
void stream_task_counts(long long row_tiles, long long pairs, int most_cs, int sms, F&& consider) {
    for (long long m = 1; m <= most_cs && row_tiles * m <= std::min<long long>(sms, pairs); ++m) consider(row_tiles * m);
    consider(std::min<long long>(sms, pairs));
}

// Up to 16 batch columns: contiguous ranges of the layers' (row tile, slice) pairs, met in the accumulate words.  tasks = 0 if
// they cannot be.  (candidate >= 0: that one of the task counts instead of the cheapest, for rabit_selftest_gemm_plan.)  (Against tasks over clusters or one per row tile: 4096 x 4096 8.6 -> 7.8 us, with one path 7.2 -> 6.5,
// 4096 x 14336 16.5 -> 15.8, 28672 x 8192 55 -> 44; nowhere slower, so such calls look no further.)
Plan stream_plan(int n_layers, const int* n_rt, const int* n_ct, int K, bool deq, int batch, int sms, int candidate = -1) {
    Plan best = {};
    Plan p = {};
    p.stream = p.split = p.max16 = p.box16 = 1;
    const int n_ops = deq ? 1 : K;
    long long pairs = 0, row_tiles = 0;
    int most_cs = 0, tail = kSliceSteps;                  // tail: steps of the shortest last slice
    bool wide_x = true;
    for (int l = 0; l < n_layers; ++l) {
        const int steps = (n_ct[l] + 1) / 2, n_cs = (steps + kSliceSteps - 1) / kSliceSteps;
        pairs += (long long)n_rt[l] * n_cs;
        row_tiles += n_rt[l];
        most_cs = std::max(most_cs, n_cs);
        if (steps % kSliceSteps != 0) tail = std::min(tail, steps % kSliceSteps);
        wide_x = wide_x && n_ct[l] % 2 == 0;
    }
    if (most_cs > RABIT_LUT_MAX_SLICES || pairs >= kMaxPairs || sms > kMaxTasks || !fill_resources(p, K, deq, tail, wide_x)) return best;
    best.clocks = 1e300;
    const double pair = kSliceSteps * (n_ops * kStreamUnit[n_ops - 1] + (deq ? (K - 1) * kStreamDeq : 0.0));
    int considered = 0;
    stream_task_counts(row_tiles, pairs, most_cs, sms, [&](long long tasks) {
        if (candidate >= 0 && considered++ != candidate) return;
        p.tasks = (int)tasks;
        double worst = 0.0;
        long long parts = 0, base = 0, t = 0;             // tasks that end in a segment that is not a whole row tile
        int l = 0;
        double c = 0.0;
        for (long long at = 0; at < pairs;) {             // segment by segment
            const int n_cs = ((n_ct[l] + 1) / 2 + kSliceSteps - 1) / kSliceSteps;
            const long long t_end = pairs * (t + 1) / tasks, tile_end = at + n_cs - (at - base) % n_cs, end = std::min(t_end, tile_end);
            c += (double)(end - at) * pair + (c > 0.0 ? kStreamPass : 0.0);
            const bool part = end - at < n_cs;
            at = end;
            if (at == base + (long long)n_rt[l] * n_cs && l + 1 < n_layers) { base = at; ++l; }
            if (at == t_end) { worst = std::max(worst, c + (part ? kStreamPublish : 0.0)); parts += part; c = 0.0; ++t; }
        }
        p.clocks = kStreamLaunch + worst + parts * 128.0 * batch / kStreamRate;
        if (p.clocks < best.clocks) best = p;
    });
    return best;
}

// (device < 0: planned without a GPU, as if it placed every cluster that its SMs have room for)
Plan make_plan(int n_rt, int n_steps, int K, bool deq, int batch, int sms, int device, bool wide_x) {
    const int n16 = (batch + kGroupCols - 1) / kGroupCols;
    const int n_ops = deq ? 1 : K;
    if (n16 == 1) {
        const int n_ct = wide_x ? 2 * n_steps : 2 * n_steps - 1;
        const Plan p = stream_plan(1, &n_rt, &n_ct, K, deq, batch, sms);
        if (p.tasks > 0) return p;
    }
    Plan best = {};
    best.clocks = 1e300;
    // (a) uniform tasks: every row tile in `chunks` chunks, the contraction of a task over `split` CTAs
    for (int chunks = 1; chunks <= n16; ++chunks) {
        Plan p = {};
        p.max16 = p.chunk16 = p.box16 = (n16 + chunks - 1) / chunks;
        p.chunks = (n16 + p.chunk16 - 1) / p.chunk16;
        if (p.chunks != chunks) continue;
        for (int seq = 0; seq <= (K == 3 && !deq ? 1 : 0); ++seq)
            for (int split = 1; split <= 8; ++split) {
                p.split = split;
                p.seq = seq;
                p.tasks = n_rt * chunks;
                const long long ctas = (long long)p.tasks * split;
                if (split > 1 && (n_steps / split < 4 || ctas > sms)) continue;
                if (!fill_resources(p, seq ? 1 : K, deq, n_steps / split, wide_x)) continue;
                if (split > 1 && device >= 0 && (prepare_kernel(K, deq, device, false, seq != 0) != cudaSuccess || resident_clusters(kernel_for(K, deq, false, seq != 0), threads_of(K, deq, seq != 0, false), split, p.smem, sms) < p.tasks)) continue;
                const double rounds = (double)((ctas + sms - 1) / sms);
                p.clocks = kLaunchClocks + (split > 1 ? kExchangeClocks * (1 + seq) : 0.0) + rounds * ((n_steps + split - 1) / split) * n_ops * unit_clocks(p.chunk16, p, seq ? 1 : n_ops) +
                           (rounds * (seq ? K : 1) - 1.0) * kPassClocks;
                if (p.clocks < best.clocks) best = p;
            }
        if (p.chunk16 <= 4) break;                   // narrower passes cost as much as these
    }
    // (b) contiguous ranges of groups, one per SM: no last wave
    const long long groups = (long long)n_rt * n16;
    if (groups >= 2LL * sms && groups < (1LL << 30)) {
        Plan p = {};
        p.split = 1;
        p.tasks = sms;
        const int per_sm = (int)((groups + sms - 1) / sms);
        for (p.max16 = std::min(16, n16); p.max16 > 1; --p.max16) {
            // most passes of a range are cut to this size: two boxes of it make one step
            const int run = std::min(per_sm, n16), pieces = (run + p.max16 - 1) / p.max16;
            p.box16 = ((run + pieces - 1) / pieces + 1) / 2;
            if (fill_resources(p, K, deq, n_steps, false)) break;
        }
        if (fill_resources(p, K, deq, n_steps, false)) {
            double worst = 0.0;
            for (int t = 0; t < sms; ++t) {
                long long g = groups * t / sms;
                const long long g1 = groups * (t + 1) / sms;
                double c = 0.0;
                while (g < g1) {
                    const int run = (int)std::min<long long>(g1 - g, n16 - g % n16), pieces = (run + p.max16 - 1) / p.max16, n = (run + pieces - 1) / pieces;
                    c += n_steps * n_ops * unit_clocks(n, p, n_ops) + kPassClocks;
                    g += n;
                }
                worst = std::max(worst, c);
            }
            p.clocks = kLaunchClocks - kPassClocks + worst;
            if (p.clocks < best.clocks) best = p;
        }
    }
    return best;
}

int sms_of(const rabit_layer& L) { return L.sm_count > 0 ? L.sm_count : 148; }

// The plan of a layer, or of several in one launch.
Plan plan_for(const rabit_layer* const* layers, int n_layers, bool deq, int batch) {
    struct Entry { int n, n_rt[kMaxGroup], n_ct[kMaxGroup], K, deq, n16, sms; Plan plan; };
    static thread_local std::vector<Entry> plans;     // a search costs tens of microseconds; a program calls few shapes
    const int n16 = (batch + kGroupCols - 1) / kGroupCols, K = layers[0]->geom.K, sms = sms_of(*layers[0]);
    for (const Entry& e : plans) {
        bool same = e.n == n_layers && e.K == K && e.deq == (int)deq && e.n16 == n16 && e.sms == sms;
        for (int l = 0; l < n_layers && same; ++l) same = e.n_rt[l] == layers[l]->geom.n_rt && e.n_ct[l] == layers[l]->geom.n_ct;
        if (same) return e.plan;
    }
    Entry e = {};
    e.n = n_layers; e.K = K; e.deq = (int)deq; e.n16 = n16; e.sms = sms;
    for (int l = 0; l < n_layers; ++l) { e.n_rt[l] = layers[l]->geom.n_rt; e.n_ct[l] = layers[l]->geom.n_ct; }
    e.plan = n_layers > 1 ? stream_plan(n_layers, e.n_rt, e.n_ct, K, deq, n16 * kGroupCols, sms)
                          : make_plan(e.n_rt[0], (e.n_ct[0] + 1) / 2, K, deq, n16 * kGroupCols, sms, layers[0]->device, e.n_ct[0] % 2 == 0);
    if (plans.size() >= 256) plans.clear();
    plans.push_back(e);
    return plans.back().plan;
}
Plan plan_for(const rabit_layer& L, bool deq, int batch) {
    const rabit_layer* one = &L;
    return plan_for(&one, 1, deq, batch);
}

void fill_layer(GemmLayer& D, const rabit_layer& L, void* y, int pair0) {
    const RabitGeom& G = L.geom;
    D.bits = reinterpret_cast<const unsigned char*>(L.d_bits);
    D.g = (const __half*)L.d_g;
    D.h = (const __half*)L.d_h;
    D.y = (__half*)y;
    D.status = L.d_status;
    D.acc = L.d_acc;
    D.M = G.M; D.N = G.N; D.Mp = G.Mp; D.n_rt = G.n_rt; D.n_ct = G.n_ct; D.n_cs = G.n_cs;
    D.fix_bits = G.fix_bits;
    D.unit = ldexpf(1.f, G.unit_exp); D.inv_unit = ldexpf(1.f, -G.unit_exp); D.limit = ldexpf(1.f, G.fix_bits);
    D.pair0 = pair0;
}
template <int NL>
void fill_common(GemmParams<NL>& P, const Plan& p, int n_layers, int batch, long long n_groups, [[maybe_unused]] int withhold) {
    P.n_layers = n_layers;
    P.batch = batch;
    P.n16 = (batch + kGroupCols - 1) / kGroupCols;
    P.n_tasks = p.tasks;
    P.chunks = p.chunks; P.chunk16 = p.chunk16;
    P.n_groups = (int)std::min<long long>(0x7FFFFFFF, n_groups);          // (only read where it fits)
    P.quot = P.n_groups / P.n_tasks; P.rem = P.n_groups % P.n_tasks;
    P.max16 = p.max16;
    P.split = p.split;
    P.recv_off = p.recv_off;
    P.stages = p.stages; P.stage_bytes = p.stage_bytes; P.x_steps = p.x_steps; P.w_stages = p.w_stages;
    P.box16 = p.box16;
    P.n_acc = p.n_acc;
    P.units = p.units; P.a_col = ((p.stream ? 2 : 1) * p.n_acc + p.seq) * p.max16 * kGroupCols;
#ifdef RABIT_CHECKED
    P.withhold = withhold;
#endif
}

// The passes of every task of a plan, kPassInts integers each; their number.
constexpr int kPassInts = 10;
template <int NL, bool SEQ>
int list_passes(GemmParams<NL>& P, const Plan& p, int n_layers, const int (*shape)[2], int K, int batch, int* out, int max_passes) {
    long long pairs = 0;
    for (int l = 0; l < NL; ++l) {
        GemmLayer& D = P.L[l];
        const int k = l < n_layers ? l : 0;
        D.N = shape[k][1];
        D.n_rt = (shape[k][0] + kTileM - 1) / kTileM;
        D.n_ct = D.N / RABIT_TILE_COLS;
        D.n_cs = (D.N + RABIT_LUT_COLS - 1) / RABIT_LUT_COLS;
        D.pair0 = (int)pairs;
        if (l < n_layers) pairs += (long long)D.n_rt * D.n_cs;
    }
    P.paths = K;
    fill_common(P, p, n_layers, batch, p.stream ? pairs : (long long)P.L[0].n_rt * ((batch + kGroupCols - 1) / kGroupCols), -1);
    int n = 0;
    for (int task = 0; task < p.tasks; ++task)
        for (int rank = 0; rank < p.split; ++rank) {
            PassWalker<NL, SEQ> w(P, task, rank);
            Pass ps;
            while (w.next(P, ps)) {
                if (n == max_passes) return -1;
                const GemmLayer& L = P.L[ps.l];
                const int arrivals = p.stream ? segment_arrivals((uint32_t)(L.pair0 + ps.rt * L.n_cs), (uint32_t)L.n_cs, (uint32_t)P.n_tasks, (uint32_t)P.n_groups) : 0;
                const int v[kPassInts] = {task, rank, ps.l, ps.rt, ps.c16, ps.n, ps.s_lo, ps.s_hi, ps.path, arrivals};
                std::copy(v, v + kPassInts, out + (size_t)kPassInts * n++);
            }
        }
    return n;
}

}  // namespace

// Host-only view of the work split (see rabit_selftest_gemm_plan).
int rabit_gemm_tc_plan(int n_layers, const int (*shape)[2], int K, bool deq, int batch, int sms, int candidate, int head[8], int* out, int max_passes) {
    if (n_layers < 1 || n_layers > kMaxGroup || K < 1 || K > RABIT_MAX_K || batch < 1 || batch > (1 << 24) || sms < 1 || sms > kMaxTasks) return -1;
    if (n_layers > 1 && (batch > kGroupCols || deq)) return -1;
    int n_rt[kMaxGroup], n_ct[kMaxGroup];
    for (int l = 0; l < n_layers; ++l) {
        if (shape[l][0] < 1 || shape[l][1] < RABIT_TILE_COLS || shape[l][1] % RABIT_TILE_COLS != 0) return -1;
        n_rt[l] = (shape[l][0] + kTileM - 1) / kTileM;
        n_ct[l] = shape[l][1] / RABIT_TILE_COLS;
    }
    const int cols = (batch + kGroupCols - 1) / kGroupCols * kGroupCols;
    if (candidate >= 0 && cols > kGroupCols) return -1;
    const Plan p = candidate >= 0 || n_layers > 1 ? stream_plan(n_layers, n_rt, n_ct, K, deq, cols, sms, candidate)
                                                  : make_plan(n_rt[0], (n_ct[0] + 1) / 2, K, deq, cols, sms, -1, n_ct[0] % 2 == 0);
    if (p.tasks < 1) return -1;
    const int h[8] = {p.tasks, p.split, p.stream, p.seq, p.max16, p.chunks, p.stages, p.n_acc};
    std::copy(h, h + 8, head);
    if (p.stream) {
        GemmParams<kMaxGroup> P = {};
        return list_passes<kMaxGroup, false>(P, p, n_layers, shape, K, batch, out, max_passes);
    }
    GemmParams<1> P = {};
    return p.seq ? list_passes<1, true>(P, p, 1, shape, K, batch, out, max_passes) : list_passes<1, false>(P, p, 1, shape, K, batch, out, max_passes);
}

// The same function that the kernel uses (see rabit_selftest_gemm_ready).
int rabit_gemm_tc_ready(bool stream, int pass_i, bool last, int* parity) {
    const Ready r = ready_of(stream, pass_i, last);
    *parity = (int)r.parity;
    return r.bar;
}

int rabit_gemm_tc_max_group() { return kMaxGroup; }

// One launch for several layers of at most 16 batch rows: equal path counts, no layer twice (it would share its accumulate words).
bool rabit_gemm_tc_group_supports(const rabit_layer* const* layers, int n_layers, int batch) {
    if (n_layers < 1 || n_layers > kMaxGroup || batch < 1 || batch > kGroupCols) return false;
    long long pairs = 0;
    for (int l = 0; l < n_layers; ++l) {
        const rabit_layer& L = *layers[l];
        if (!rabit_gemm_tc_supports(L, batch) || L.geom.K != layers[0]->geom.K || L.geom.n_cs > RABIT_LUT_MAX_SLICES) return false;
        pairs += (long long)L.geom.n_rt * L.geom.n_cs;
        for (int m = 0; m < l; ++m)
            if (layers[m] == &L) return false;
    }
    return pairs < kMaxPairs && sms_of(*layers[0]) <= kMaxTasks;
}

// A stream launch: the plan's contiguous ranges over the layers.
static cudaError_t launch_stream(const rabit_layer* const* layers, int n_layers, const void* const* xs, void* const* ys, int batch, bool dequantised, const Plan& p, cudaStream_t stream) {
    const int K = layers[0]->geom.K, device = layers[0]->device;
    GemmParams<kMaxGroup> P;
    P.paths = K;
    XMaps<kMaxGroup> maps;
    int pairs = 0;
    for (int l = 0; l < kMaxGroup; ++l) {
        if (l >= n_layers) { P.L[l] = P.L[0]; maps.map[l] = maps.map[0]; continue; }
        const RabitGeom& G = layers[l]->geom;
        cudaError_t e = x_tensor_map(xs[l], G.N, batch, 1, p.x_steps, &maps.map[l]);
        if (e != cudaSuccess) return e;
        fill_layer(P.L[l], *layers[l], ys[l], pairs);
        pairs += G.n_rt * G.n_cs;
    }
    fill_common(P, p, n_layers, batch, pairs, layers[0]->withhold);
    cudaError_t e = prepare_kernel(K, dequantised, device, true);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned int)p.tasks);
    cfg.blockDim = dim3((unsigned int)threads_of(K, dequantised, false, true));
    cfg.dynamicSmemBytes = p.smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    void* args[2] = {&P, &maps};
    return cudaLaunchKernelExC(&cfg, kernel_for(K, dequantised, true), args);
}

cudaError_t rabit_launch_gemm_tc_group(const rabit_layer* const* layers, int n_layers, const void* const* xs, void* const* ys, int batch, cudaStream_t stream) {
    if (n_layers == 1) return rabit_launch_gemm_tc(*layers[0], xs[0], ys[0], batch, stream);
    if (!rabit_gemm_tc_group_supports(layers, n_layers, batch)) return cudaErrorInvalidValue;
    const Plan p = plan_for(layers, n_layers, false, batch);
    if (p.tasks < 1) return cudaErrorInvalidValue;
    return launch_stream(layers, n_layers, xs, ys, batch, false, p, stream);
}

bool rabit_gemm_tc_supports(const rabit_layer& L, int batch) {
    return batch >= 1 && batch <= (1 << 24) && L.geom.K <= 3 && encode_tiled_fn() != nullptr;
}

// Estimated duration (us) of the exact-expansion GEMM on B200, at 1.9 GHz.
double rabit_gemm_tc_estimate_us(const rabit_layer& L, int batch) { return plan_for(L, false, batch).clocks / 1900.0; }

cudaError_t rabit_launch_gemm_tc(const rabit_layer& L, const void* x, void* y, int batch, cudaStream_t stream, bool dequantised) {
    const RabitGeom& G = L.geom;
    const Plan p = plan_for(L, dequantised, batch);
    if (p.tasks < 1) return cudaErrorInvalidValue;
    if (p.stream) {
        const rabit_layer* one = &L;
        return launch_stream(&one, 1, &x, &y, batch, dequantised, p, stream);
    }
    XMaps<1> maps;
    cudaError_t e = x_tensor_map(x, G.N, batch, p.box16, p.x_steps, &maps.map[0]);
    if (e != cudaSuccess) return e;
    e = prepare_kernel(G.K, dequantised, L.device, false, p.seq != 0);
    if (e != cudaSuccess) return e;

    GemmParams<1> P;
    P.paths = G.K;
    fill_layer(P.L[0], L, y, 0);
    fill_common(P, p, 1, batch, (long long)G.n_rt * ((batch + kGroupCols - 1) / kGroupCols), L.withhold);

    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned int)(p.tasks * p.split));
    cfg.blockDim = dim3((unsigned int)threads_of(G.K, dequantised, p.seq != 0, false));
    cfg.dynamicSmemBytes = p.smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = (unsigned int)p.split;
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = p.split > 1 ? 2 : 1;
    void* args[2] = {&P, &maps};
    return cudaLaunchKernelExC(&cfg, kernel_for(G.K, dequantised, false, p.seq != 0), args);
}
