// ngdbf_kernels.cuh -- shared device code of the NGDBF decoder (sm_103a): job and launch
// descriptors, the shared-memory layout and the persistent slot loop for one job.
//
// Work decomposition.  A CTA owns 32 frame slots, one per bit of a 32-bit
// word: the decisions x_k of its 32 frames are one word per symbol k and the
// syndromes s_i one word per check i (bit f set <=> x_k = -1 / check i
// unsatisfied for slot f).  Each round the CTA
//   A. forms every syndrome word as the XOR of the d_c decision words of a
//      check (Sec. III-A, Step 1 of Sec. III-B), OR-reduces them to the
//      "some check unsatisfied" mask with warp reductions,
//   B. retires slots whose frame satisfied every check (pass) or reached T
//      (smoothed output, Sec. III-E), writes their outputs, takes new frames
//      from a global atomic queue for them and loads those frames,
//   A'. adds, per symbol, the unsatisfied-check words of M(k) lane-wise (2-bit
//      lanes, three checks at a time, widened to 4-bit counts; bit-sliced for
//      symbol degrees above 15) into the count of unsatisfied checks, then
//   C. runs Step 2 / Step 3b for every symbol of every live slot: each lane draws
//      the Philox outputs of one slot's four symbols and compares each with a cutoff
//      that no flip can exceed (see "Lazy evaluation"); the few outputs at or below
//      it are queued and only for those E_k = x_k y_k + w S_k + q_k is formed and
//      compared with theta lambda^{u_k} (Step 3a: with the slot's least so far).  Symbol
//      degrees above 15 form E_k for every symbol, with lane = slot, and so do iterations in
//      which about a sixth of the outputs or more would be evaluated (full_rounds).
// When an iteration flipped few decisions (at most kFlips, a code not split over a cluster),
// A and A' are replaced by
//   D. per flip, its d_v checks toggled for the slot, the slot's number of unsatisfied checks
//      and the counts of the checks' symbols moved by one.
// Slots therefore iterate independently (each frame has its own t), a
// converged frame frees its slot at once, and the CTA only stops when the
// queue is empty and its last slot finished.
//
// Per-(symbol, slot) state: one byte of quantized margin (global scratch, L2-resident; while every
// E_k is formed the held sample is there instead), and a 16-bit word holding the flips of the symbol
// so far (bits 0-8; u_k = t - flips) and the number of -1 decisions the smoothing window will
// have seen at T if the symbol flips no more (bits 9-15), in shared memory when it fits, else
// in global scratch.  Both change only when a symbol flips.  Both are laid out by groups of
// four symbols, [k/4][slot][k%4], so that phase C reads one word per lane for the four symbols
// of a Philox call; the counts likewise, and the decision words are contiguous.  Decision and
// syndrome words, counts, the threshold and generator tables live in shared memory, the
// adjacency tables there when they fit.
//
// Lazy evaluation.  A symbol flips only when E_k < theta_k, that is when its perturbation is
// below -(x_k y_k + w S_k - theta_k); with z monotone in the Philox output r (r < 2^31 gives
// the negative deviates, in increasing order) that is r below a cutoff of the margin alone.
// Per slot the margin is kept in steps of Job::pf: a byte holds x_k y_k + w d_k - theta_hi
// rounded down, theta_hi the largest threshold the symbol can reach; w S_k = w d_k - 2 w c
// subtracts pf_K steps per unsatisfied check (one multiply for the four bytes of a group),
// and the lanes of a slot at iteration t add D(t), theta_hi - theta(t) in steps rounded down
// (theta lambda^u <= theta(t) for u <= t).  A 256-entry table maps the byte to the cutoff,
// rounded up.  Every rounding errs towards evaluating E_k, so the decisions are those of the
// dense form bit for bit; the exact form runs for the symbols at or below the cutoff only.
//
// What bounds it (one GB300, the (6,32) code of 2048 symbols, 32 live slots): a step of phase C --
// four symbols of 32 slots -- takes 75 instructions, 40 of them Philox, and 31 cycles of an SM; the
// 18 wide multiplies alone take 19 (1.05 cycles each), the ALU pipe 18, so the step is near the
// issue and pipe limits (issue 62-68 %, ALU 57-61 % busy).  Forming E_k for every symbol took 103
// cycles a step.  100003 frames at 4.5 dB (8-bit samples): 30.6 -> 12.5 ms; 200000 frames at 3.5 dB,
// where 3 % of the outputs are evaluated and A and A' run every iteration: 260 -> 193 ms.  With
// few slots an iteration is latency: 3.5 us for one frame of the (3,6) code of 1008 symbols.
//
// The single-bit variant (Step 3a) needs the least E_k of a slot: it sweeps with a guess tau, the
// slot's previous least E_k plus kGuess of its noise, in the place of the threshold.  A least
// E_k at or below tau is the slot's (every symbol that could be as low was evaluated); the
// slots without one are swept again with tau raised, at last with every symbol evaluated.
#pragma once

#include <cooperative_groups.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>
#include <type_traits>

#include "../../include/ngdbf.h"
#include "ngdbf_device.cuh"

namespace ngdbf {

constexpr int kSlots = 32;

// Symbols rounded up to whole groups of four (the per-slot arrays are laid out by groups).
__host__ __device__ inline int pad4(int n) { return (n + 3) & ~3; }
// Index of the j-th symbol of N(i): units of four (one 8-byte load), two units per check side by
// side for the two threads that share it, [j/8][i][(j/4)%2][j%4].
__host__ __device__ inline size_t chk_index(int j, int i, int m) {
    return (((size_t)(j >> 3) * m + i) * 2 + ((j >> 2) & 1)) * 4 + (j & 3);
}
__host__ __device__ inline int chk_entries(int m, int dc_max) { return m * 8 * ((dc_max + 7) >> 3); }
// Index of (symbol k, slot f) in the group layout [k/4][slot][k%4].
__host__ __device__ inline int gidx(int k, int f) { return (((k >> 2) * kSlots + f) << 2) | (k & 3); }
constexpr int kTabChk = 1;              // N(i) table in shared memory
constexpr int kTabSym = 2;              // M(k) table and degrees in shared memory
// The longest codes (without their state in shared memory): the warps' queues lie over the syndrome
// words, which phase C does not read, and flips are not recorded (no D).  Blocks of as many threads
// as there are words for queues, kTightThreads at least (4864 frames of n = 10950, m = 300, T = 60:
// 21.3 ms with 4 warps, 7.0 with 16).
constexpr int kTight = 4;
constexpr int kTightThreads = 128;

constexpr int kMaxT = NGDBF_MAX_T;
constexpr uint32_t kUMask = 0x1FFu;   // flips of the symbol so far: bits 0-8
constexpr int kCShift = 9;            // smoothing count: bits 9-15
constexpr int kNarrowDegree = 15;     // largest symbol degree of the 4-bit counts

// Lazy evaluation: margin byte kMargin0 is a margin of zero (at or below it every output is
// evaluated), pf_K d_v is at most kMarginCounts and pf_K d_v + D(t) at most kMargin0, so that
// no byte of a group borrows from or carries into another.
constexpr int kMargin0 = 96, kMarginCounts = 80;
// Most flips of one iteration of a CTA by which the syndromes and counts are moved (D).
constexpr int kFlips = 256;
// Bytes readable past a CTA's margin bytes (the last step of phase C reads whole warps of groups).
constexpr int kMarginSlack = 32 * 32 * 4;
constexpr int kQueue = 64;            // groups queued per warp for the exact form
constexpr int kCutBytes = 256 * 4;    // one cutoff table
// Outputs evaluated per group of 32 slots (of 128) in one iteration, looked at in every fourth, above which
// every E_k is formed from the next one on (full_rounds).  The exact form takes about 125 cycles of an SM
// per 32 outputs, forming every E_k about 75 cycles more than the sweep per group, so the two meet near a
// sixth of the outputs: between 2.0 and 2.5 dB for the (3,6) code of 1008 symbols (12 and 20 measured alike).
constexpr int kFullMarks = 16, kFullEvery = 3;
// What a shared-memory layout is for (smem_layout): one job per launch, a job of a table, or a
// serving CTA with cutoff tables for every chain entry (kTable + c: for c of them).
constexpr int kLaunch = 0, kTable = 1, kServe = kTable + 8;
// Single-bit: the least E_k is guessed kGuess noise scales above the last, the first kFirst above
// the lowest tau followed, raised by kRaise at a time and to infinity after kSweeps sweeps.
constexpr float kGuess = 1.5f, kFirst = 2.0f, kRaise = 2.0f;
constexpr int kSweeps = 5;

// Arithmetic of the held samples and of E_k (Sec. IV-E): the perturbation is
// always the FP32 generator output.
enum Precision { kFP32 = 0, kFP16 = 1, kFIX = 2, kFIXACC = 3 };
constexpr int kAccBits = 8;           // FIXACC: accumulator steps per half level = 2^8

template <int PREC> struct Held;
template <> struct Held<kFP32> { using T = float; };
template <> struct Held<kFP16> { using T = __half; };
template <> struct Held<kFIX> { using T = int8_t; };      // signed level code b, value 2b + 1
template <> struct Held<kFIXACC> { using T = int8_t; };   // the same Eq. 8 level code

// Slot scratch of CTA `cta` of a launch whose CTAs hold n symbols each: room for a held sample per
// (symbol, slot), whose first part the margin bytes take.
template <int PREC>
__device__ __forceinline__ typename Held<PREC>::T* slot_scratch(void* base, int cta, int n) {
    return static_cast<typename Held<PREC>::T*>(base) + (size_t)cta * pad4(n) * kSlots;
}

// One decode job: a code, a batch of frames and the parameters of the method.
struct Job {
    // code tables (device)
    int32_t n, m, dv_max, dc_max;
    const uint16_t* chk_cols;   // N(i), chk_index layout, padded with n
    const uint16_t* sym_chks;   // M(k), [dv_max][ceil(n / 4)][4], padded with m
    const uint8_t* sym_deg;     // [n]           d_v(k)
    // batch
    const float* y;             // [n_frames][n]
    int64_t n_frames;
    uint64_t frame_offset;
    uint8_t* bits;              // [n_frames][nb]
    int32_t* iters;
    uint8_t* pass;
    int32_t nb;
    // parameters
    float w, scale, y_max;      // w: FP32 value, or its binary16 value for FP16
    int32_t clamp, t_max, t_smooth;   // t_smooth = max(0, T - W)
    float fix_R;                // fixed point: fl32(2^Q / (2 Y_max)), kmax = 2^(Q-1) - 1, W~
    int32_t fix_kmax, fix_W;
    float acc_R;                // FIXACC: accumulator steps per unit fl32(2^(Q+8) / Y_max), w in steps
    int32_t acc_W;
    // lazy evaluation (see the top; real units are those of y): steps per unit, w in steps, the
    // byte of x_k y_k + w d_k = 0, the byte's range, D(t) = floor(pf_d0 - pf_d1 theta(t)) <=
    // pf_dcap with theta(t) as held in thr (single-bit: the shift floor(pf_d0 - pf_d1 tau) <= 0
    // of the byte, its zero margin at the lowest tau followed), real value of one integer unit
    // (fixed point) or 1, steps per unsatisfied check, the step in units of `scale`
    // (rounded down), and single-bit: the lowest tau followed
    float pf_inv, pf_w, pf_bias, pf_lo, pf_hi, pf_d0, pf_d1, pf_unit, pf_rho, pf_low;
    int32_t pf_K, pf_dcap;
    int32_t slots;              // frames a CTA takes first (1..32): the batch spread over the launch (serving: 32)
    // thresholds theta lambda^u, u = 0..T: FP32 bits, binary16 values as FP32 bits, or
    // fixed-point levels Theta~(u) (FIX) or steps (FIXACC) as int32 (device memory; the
    // single-job launch passes them inline instead)
    const uint32_t* thr;
    unsigned long long* queue;  // next unclaimed frame of this job
    long long work;             // job tables: estimated work of one frame, n x (T + 1)
    int32_t single;             // Step 3a: flip only the symbol with the least E_k (ties: lowest k)
    int32_t uniform;            // Sec. V-B: uniform perturbation of the same variance
    // objective trace of frames 0 .. trace_frames-1 (nullptr: off): unsatisfied checks U(t) and
    // the correlation C(t) = sum_k rint(x_k y~_k 2^32), [frame][t_max + 1]
    int32_t* trace_u;
    long long* trace_c;
    long long trace_frames;
    double trace_yunit;         // FIX / FIXACC: value of one half level, Y_max 2^-Q
    // serving (0 / nullptr otherwise): `queue` holds (gen << 32) | frames claimed and claims
    // check the generation, so a CTA still holding an earlier job of the same ring slot never
    // takes frames of a later one; the CTA that finishes the last frame counts it in `done` and
    // writes `gen` into the host-visible word `notify`
    uint32_t gen;
    unsigned int* done;
    unsigned int* notify;
    const unsigned int* retire;     // serving: nonzero once the resident kernel is retiring (no claims)
    // serving: jobs with the same nonzero chain_key have the same code and decoding parameters
    // (they differ only in samples, sigma, frame offset, outputs and counters), so a CTA may
    // decode frames of several of them in its slots at once
    unsigned long long chain_key;
    // launches of one job (nullptr otherwise): the frames in the slots of all such launches on the
    // device, and the CTAs that can be resident (see busy_slots)
    unsigned int* in_flight;
    int32_t cap;
};

// Chaining of serving jobs inside one CTA (decode_job with CHAIN): the jobs whose frames the
// slots hold (entries of jl, slot f holds a frame of jl[slot_e[f]]), the entry frames are
// claimed from, and `next`, which finds another published job with the same chain_key.
constexpr int kChain = 8;
static_assert(kServe == kTable + kChain, "a cutoff table per chain entry");
struct NoNext {
    __device__ bool operator()(unsigned long long, Job&) const { return false; }
};
template <class Next>
struct ChainCtx {
    Job* jl;                    // [kChain] shared memory
    int8_t* slot_e;             // [kSlots] shared memory
    int* cur_e;                 // shared memory
    Next next;
    int entries;                // entries in use: kChain, or the cutoff tables of the layout when fewer
};

// Static shared memory of the serving kernel.
struct ServeShared {
    Job jl[kChain];             // [0]: the request picked; the others: chained requests
    unsigned long long fail[2];
    int8_t slot_e[kSlots];
    int cur_e, pick;
};

// Claims up to k consecutive frames of job A: returns true and the first frame id in *base
// (ids at or beyond A.n_frames mean no frame), or false when none is left.  Serving jobs
// (A.gen != 0) claim by compare-and-swap within their generation, at most kClaimTries times.
constexpr int kClaimTries = 4096;
__device__ __forceinline__ bool claim_frames(const Job& A, unsigned k, unsigned long long* base) {
    if (A.gen == 0u) {
        *base = atomicAdd(A.queue, (unsigned long long)k);
        return true;
    }
    // a retiring resident kernel takes no new frames: they wait for the next launch, which
    // has every CTA, instead of being decoded by the few CTAs still finishing
    if (A.retire != nullptr && *(const volatile unsigned int*)A.retire != 0u) return false;
    unsigned long long old = *(volatile unsigned long long*)A.queue;
    for (int it = 0; it < kClaimTries; ++it) {
        if ((uint32_t)(old >> 32) != A.gen || (long long)(uint32_t)old >= A.n_frames) return false;
        const unsigned long long got = atomicCAS(A.queue, old, old + k);
        if (got == old) {
            *base = (uint32_t)old;
            return true;
        }
        old = got;
    }
    return false;
}

// Frames a CTA takes first of job A: A.slots, unless other launches have frames on the device.  A launch
// by itself is fastest spread over every CTA, but a frame then costs up to six times the SM time of one
// among 32, so launches that share the device pack their frames: twice as densely as those in flight and
// the launch's own would lie over all CTAs, which leaves CTAs for launches to come, and comes to 32 a CTA
// within a few generations of launches on a full device.  64 streams of 96 frames of the (6,32) code of
// 2048 symbols at 3.0 dB, 256 calls: 62 ms packed by 32, 252 spread, 55 so; one such call by itself 1.4 ms
// at 4.0 dB (7.3 packed).  (The launch's own frames in flight are at most those claimed from its queue, read
// after the total: by itself it sees no others.)
__device__ __forceinline__ unsigned busy_slots(const Job& A) {
    if (A.in_flight == nullptr || A.slots >= kSlots || A.n_frames == 1) return (unsigned)A.slots;
    const unsigned all = *(volatile unsigned int*)A.in_flight, own = (unsigned)*(volatile unsigned long long*)A.queue;
    if (all <= own) return (unsigned)A.slots;
    // (fewer than 32 frames for each CTA: a small number)
    const unsigned k = (2u * (all - own + (unsigned)A.n_frames) + (unsigned)A.cap - 1u) / (unsigned)A.cap;
    return min(max(k, (unsigned)A.slots), (unsigned)kSlots);
}

// Offsets in bytes of the shared-memory arrays (smem_layout).
struct SmemLayout {
    int32_t off_frame, off_start, off_ctl, off_unsat, off_flips, off_best, off_tau, off_trace, off_icdf, off_cut, off_queue, off_xw, off_sw, off_cnt,
        off_thr, off_st, off_chk, off_sym, cuts, total;
};

// Launch of one job: the job and its thresholds travel as kernel parameters.
struct DecodeArgs {
    Job J;
    int32_t placement;          // adjacency tables copied into shared memory: kTabChk | kTabSym
    void* yslots;               // [grid][pad4(n)/4][32][4] margin bytes, or held samples of 4, 2 or 1 bytes
    uint16_t* st_global;        // [grid][pad4(n)/4][32][4] when the state is not in shared memory
    SmemLayout L;
    GenConsts G;
    uint32_t thr[kMaxT + 1];
};

// Launch of a job table: CTA c starts with job first_job[c] and, once that job has
// no unclaimed frame left and its slots are idle, moves to the job with the most
// unclaimed work (frames x Job::work).  Each job gets its own shared-memory layout
// (job_layout); the launch has room for the largest.
struct MultiArgs {
    const Job* jobs;
    int32_t n_jobs;
    const int32_t* first_job;   // [grid]
    const int32_t* slots;       // [n_jobs] Job::slots under this launch shape
    int32_t n_max, m_max, t_max, dv_max, dc_max;   // layout maxima over the jobs
    int32_t placement;          // adjacency tables copied into shared memory: kTabChk | kTabSym
    // cluster launches: jobs with n >= split_min_n are split over the `cluster` CTAs of a
    // cluster (n_local symbols per CTA at most); the per-CTA arrays hold n_local symbols
    int32_t cluster, split_min_n, n_local;
    int32_t smem_bytes;         // dynamic shared memory of the launch (every job's layout fits)
    void* yslots;               // [grid][pad4(n_local)/4][32][4]
    uint16_t* st_global;        // [grid][pad4(n_local)/4][32][4] when the state is not in shared memory
    GenConsts G;
};

// Symbols one CTA decodes when the `size` CTAs of a cluster share one 32-slot group: [k_lo, k_hi),
// k_lo a multiple of 32 (size 1: the whole code).  Rank r of C takes chunks of 32 symbols
// [r nc / C, (r + 1) nc / C) of the nc = ceil(n / 32) chunks.
struct Split {
    int rank, size, k_lo, k_hi;
};
__host__ __device__ inline Split split_range(int rank, int size, int n) {
    const int nc = (n + 31) / 32;
    Split S;
    S.rank = rank;
    S.size = size;
    S.k_lo = 32 * (rank * nc / size);
    S.k_hi = 32 * ((rank + 1) * nc / size);
    if (S.k_hi > n) S.k_hi = n;
    return S;
}
// Largest number of symbols a CTA holds when a code of n symbols is split over `size` CTAs.
__host__ __device__ inline int split_local_max(int n, int size) { return 32 * (((n + 31) / 32 + size - 1) / size); }


// Offsets in bytes of the shared-memory arrays (-1: not placed).  ctl holds: [0..1] unsatisfied
// masks (double-buffered by pass parity; wide and split jobs), [2] live mask, [3] new-slot
// mask, [4] chain entries loaded (launches of one job: the frames taken first), [5] single-bit slots left, [6..7] flips of this iteration
// (double-buffered by round parity).
// When d_v <= 15 (narrow), sw holds per check two words with one 2-bit lane per slot (lane
// f & 15 of word f >> 4: 1 when check i is unsatisfied for slot f), and cnt holds per group of
// four symbols sixteen words of their counts of unsatisfied checks: byte k % 4 of word
// cnt_word(f), nibble cnt_shift(f) (16 bytes per symbol).  Otherwise (wide) sw holds
// the 32-bit unsatisfied mask of each check and cnt, per symbol, the bit-sliced count
// (seven words, bit f for slot f) and d_v(k) (32 bytes).  xw has room for whole groups
// and the zero sentinel word at index n.
// `wide` (< 0: from dv_max) selects the count and syndrome formats, which follow the kernel's
// WIDE template argument when a job table lays out a job of lower degree.
// `use`: a launch of one job, a job of a table (no objective trace), or kServe cutoff tables of
// a serving CTA, one per chain entry (no trace, and no second buffer of the single-bit minima,
// which only CTAs of a cluster use).
__host__ __device__ inline SmemLayout smem_layout(int n, int m, int t_max, int dv_max, int dc_max,
                                                  bool need_thr, bool st_smem, int tables, int n_local = -1,
                                                  int wide = -1, int use = kLaunch, int tight_warps = kTightThreads / 32) {
    if (n_local < 0) n_local = n;   // symbols whose counts, state and M(k) rows this CTA holds
    const bool wd = wide < 0 ? dv_max > kNarrowDegree : wide != 0;
    SmemLayout L;
    int o = 0;
    auto take = [&](int bytes, int align) {
        o = (o + align - 1) / align * align;
        int r = o;
        o += bytes;
        return r;
    };
    const int cnt_bytes = wd ? 32 : 16;
    L.off_frame = take(kSlots * 8, 16);
    L.off_start = take(kSlots * 4, 16);
    L.off_ctl = take(8 * 4, 16);
    const bool tight = (tables & kTight) != 0;
    // (wide: none of the lazy form's arrays)
    L.off_unsat = wd ? -1 : take(kSlots * 4, 16);   // number of unsatisfied checks of each slot
    const int serve = use > kTable ? use - kTable : 0;      // cutoff tables asked for
    L.off_best = take((serve ? 1 : 2) * kSlots * 8, 16);    // single-bit variant: least (E key, k) per slot, two rounds
    L.off_tau = wd ? -1 : take(kSlots * 4, 16);     // single-bit variant: guess of each slot's least E_k
    L.off_trace = use == kLaunch ? take(kSlots * 12, 16) : -1;  // objective trace: per slot C (int64), then U (int32)
    L.off_icdf = take(256 * 16, 16);       // inverse normal CDF coefficients
    L.cuts = wd ? 0 : serve ? serve : 1;
    L.off_cut = wd ? -1 : take(L.cuts * kCutBytes, 16);     // cutoff of each margin byte
    L.off_cnt = take(pad4(n_local) * cnt_bytes, 16);
    L.off_flips = wd || tight ? -1 : take(kFlips * 4, 16);   // flips of this iteration: local symbol | slot << 16
    // per warp: groups for the exact form (phase C's last steps may read up to 31 groups of counts
    // past the code's: they lie inside this array)
    L.off_queue = wd || tight ? -1 : take(32 * kQueue * 4, 16);
    L.off_xw = take(pad4(n + 1) * 4, 16);
    const int sw_bytes = (m + 1) * (wd ? 4 : 8), queues = tight_warps * kQueue * 4;
    L.off_sw = take(tight && sw_bytes < queues ? queues : sw_bytes, 16);
    if (tight) L.off_queue = L.off_sw;
    // all 512 values of the 9-bit u field: an idle slot's counter may pass T (its lookups are
    // don't-care but stay inside the table)
    L.off_thr = need_thr ? take((kUMask + 1) * 4, 16) : -1;
    L.off_st = st_smem ? take(pad4(n_local) * kSlots * 2, 16) : -1;
    L.off_chk = (tables & kTabChk) ? take(chk_entries(m, dc_max) * 2, 16) : -1;
    L.off_sym = (tables & kTabSym) ? take(pad4(n_local) * dv_max * 2 + pad4(n_local), 16) : -1;
    L.total = (o + 15) / 16 * 16;
    return L;
}

// Layout L of a narrow or wide kernel with the offsets that do not depend on the code (all up to
// the counts, or of a serving CTA to the cutoff tables) as compile-time constants.
template <bool WIDE, int USE = kLaunch>
__device__ __forceinline__ SmemLayout with_fixed_offsets(SmemLayout L) {
    const SmemLayout F = smem_layout(4, 1, 0, 1, 1, false, false, 0, -1, WIDE ? 1 : 0, USE);
    L.off_frame = F.off_frame;
    L.off_start = F.off_start;
    L.off_ctl = F.off_ctl;
    L.off_unsat = F.off_unsat;
    L.off_best = F.off_best;
    L.off_tau = F.off_tau;
    L.off_trace = F.off_trace;
    L.off_icdf = F.off_icdf;
    L.off_cut = F.off_cut;
    if (USE <= kTable) L.off_cnt = F.off_cnt;
    return L;
}

// Layout of one job of a job table: arrays sized for the job's own code (n_local symbols per
// CTA: its share when split over a cluster) in the launch's count and syndrome format, with
// as many of the adjacency tables that `tables` allows as fit in `bytes` (both, then N(i)
// alone, M(k) alone, none, then kTight without state); *tables_out receives the placement taken.
// A serving job (use > kTable) has a cutoff table for every chain entry if it fits so in any
// of these ways but kTight; else for as many as fit, one at least.  `warps`: of the block, each with
// its queue.  Host planning and the kernel evaluate it alike, so the launch's shared memory is the largest job's, not the layout of
// the table's maxima.
__host__ __device__ inline SmemLayout job_layout(int n, int m, int t_max, int dv_max, int dc_max, bool need_thr,
                                                 bool st_smem, bool wide, int tables, int n_local, int bytes,
                                                 int* tables_out, int use = kTable, int warps = kTightThreads / 32) {
    const int opts[5] = {tables & (kTabChk | kTabSym), tables & kTabChk, tables & kTabSym, 0, kTight};
    const bool serve = use > kTable;
    SmemLayout L{};
    auto place = [&](int u, int n_opts) {
        for (int i = 0; i < n_opts; ++i) {
            L = smem_layout(n, m, t_max, dv_max, dc_max, need_thr, st_smem, opts[i], n_local, wide ? 1 : 0, u, warps);
            *tables_out = opts[i];
            if (L.total <= bytes) return true;
        }
        return false;
    };
    // (with its state in shared memory only if every chain entry fits too)
    if (!place(use, wide || st_smem || serve ? 4 : 5) && serve && !wide && !st_smem) place(kTable + 1, 5);
    if (serve && L.cuts > 0 && L.total <= bytes) {       // the room left: more of the cutoff tables
        const int more = (bytes - L.total) / kCutBytes, want = use - kTable - L.cuts;
        L = smem_layout(n, m, t_max, dv_max, dc_max, need_thr, st_smem, *tables_out, n_local, 0,
                        kTable + L.cuts + (more < want ? more : want), warps);
    }
    return L;
}

// Signed fixed-point level code of v (Eq. 8): k = min(floor(|v| R), kmax) decided in FP32,
// b = k for v >= 0 and -k - 1 otherwise; the level's value is 2b + 1 in units of Delta/2.
__host__ __device__ inline int32_t fix_code(float v, float R, int32_t kmax) {
#ifdef __CUDA_ARCH__
    const float a = __fmul_rn(fabsf(v), R);
    const int32_t k = (a < (float)kmax) ? __float2int_rd(a) : kmax;
#else
    const float a = std::fabs(v) * R;
    const int32_t k = (a < (float)kmax) ? (int32_t)std::floor(a) : kmax;
#endif
    return v >= 0.0f ? k : -k - 1;
}

// Order-preserving 32-bit key of an FP32 value (-0 counts as +0, as a comparison would).
__device__ __forceinline__ uint32_t order_key(float v) {
    uint32_t b = __float_as_uint(v);
    if (b == 0x80000000u) b = 0u;
    return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}

// Bits 0..15 of b moved to bits 0, 2, ..., 30 (one bit per 2-bit lane).
__device__ __forceinline__ uint32_t spread_pairs(uint32_t b) {
    b = (b | (b << 8)) & 0x00FF00FFu;
    b = (b | (b << 4)) & 0x0F0F0F0Fu;
    b = (b | (b << 2)) & 0x33333333u;
    return (b | (b << 1)) & 0x55555555u;
}

// Word of a group's sixteen count words, and bit offset in each of its four bytes, that hold
// slot f (what widening 2-bit lanes to even and odd nibbles and gathering bytes gives).
__device__ __forceinline__ int cnt_word(int f) { return ((f >> 4) << 3) | ((f & 1) << 2) | ((f >> 2) & 3); }
__device__ __forceinline__ int cnt_shift(int f) { return (f & 2) << 1; }

// Position of the (j+1)-th set bit of mask (j < popc(mask)), by halving.
__device__ __forceinline__ int select_bit(uint32_t mask, int j) {
    int pos = 0;
#pragma unroll
    for (int w = 16; w; w >>= 1) {
        const int c = __popc(mask & ((1u << w) - 1u));
        if (j >= c) {
            j -= c;
            mask >>= w;
            pos += w;
        }
    }
    return pos;
}

// Lane f receives the number of lanes whose word has bit f set (a 32 x 32 bit transpose).
__device__ __forceinline__ int column_count(uint32_t s, int lane) {
    uint32_t mask = 0x0000FFFFu;
#pragma unroll
    for (int j = 16; j; j >>= 1) {
        const uint32_t t = __shfl_xor_sync(0xFFFFFFFFu, s, j);
        s = (lane & j) ? (s & ~mask) | ((t & ~mask) >> j) : (s & mask) | ((t & mask) << j);
        mask ^= mask << (j >> 1);
    }
    return __popc(s);
}

// Position of the (j+1)-th set bit of mask (j < popc(mask)).
__device__ __forceinline__ int nth_set_bit(uint32_t mask, int j) {
    for (int i = 0; i < j; ++i) mask &= mask - 1u;
    return __ffs(mask) - 1;
}

// The held form of a channel sample: saturated, then rounded or quantized (Sec. IV-A, IV-E).
template <int PREC>
__device__ __forceinline__ typename Held<PREC>::T hold(float v, const Job& A) {
    if (A.clamp) {
        if (v > A.y_max) v = A.y_max;
        if (v < -A.y_max) v = -A.y_max;
    }
    if constexpr (PREC == kFP32) return v;
    else if constexpr (PREC == kFP16) return __float2half_rn(v);
    else return (int8_t)fix_code(v, A.fix_R, A.fix_kmax);
}
// x(0) = sign(y): whether the held sample is negative (sign(-0) = +1).
template <int PREC>
__device__ __forceinline__ bool held_negative(typename Held<PREC>::T h) {
    if constexpr (PREC == kFP32) return !(h >= 0.0f);
    else if constexpr (PREC == kFP16) return !(__half2float(h) >= 0.0f);
    else return h < 0;
}
// Sample f of job A at symbol k (a serving job's samples are read past L1).
__device__ __forceinline__ float read_sample(const Job& A, long long frame, int k) {
    const float* p = A.y + (size_t)frame * A.n + k;
    return A.gen ? __ldcg(p) : __ldg(p);
}

// E_k = ((x_k y_k) + w S_k) + q_k in the arithmetic of PREC, rounded after every operation
// (Step 2): FP32 and FP16 give it as an FP32 value, the fixed-point forms as an integer.
template <int PREC> struct Metric { using T = int32_t; };
template <> struct Metric<kFP32> { using T = float; };
template <> struct Metric<kFP16> { using T = float; };
// (S is an integer or the float of the same value.)
__device__ __forceinline__ float as_float(int S) { return __int2float_rn(S); }
__device__ __forceinline__ float as_float(float S) { return S; }
// What metric() takes from a job.
struct MetricConsts {
    float w, fix_R;
    int32_t fix_kmax, fix_W;
    float acc_R;
    int32_t acc_W;
};
template <int PREC, class Sum, class Consts>
__device__ __forceinline__ typename Metric<PREC>::T metric(typename Held<PREC>::T h, uint32_t xsign, Sum S, float q,
                                                           const Consts& A) {
    if constexpr (PREC == kFP32) {
        const float xy = __uint_as_float(__float_as_uint(h) ^ xsign);
        return __fadd_rn(__fadd_rn(xy, __fmul_rn(A.w, as_float(S))), q);
    } else if constexpr (PREC == kFP16) {
        // fl(w S_k) is the exact product of a binary16 w and a small integer; the additions are
        // binary16 additions (a correctly rounded FP32 addition of binary16 operands rounded
        // once more to binary16 gives the same value)
        const __half xy = __ushort_as_half(__half_as_ushort(h) ^ (uint16_t)(xsign >> 16));
        const float ws = __fmul_rn(A.w, as_float(S));
        return __half2float(__hadd(__hadd(xy, __float2half_rn(ws)), __float2half_rn(q)));
    } else if constexpr (PREC == kFIX) {
        // Eq. 9 in units of Delta/2, exact integers
        const int32_t Y = 2 * (int32_t)h + 1;
        const int32_t Qv = 2 * fix_code(q, A.fix_R, A.fix_kmax) + 1;
        return (xsign ? -Y : Y) + A.fix_W * S + Qv;
    } else {
        // the held Eq. 8 level in accumulator steps (2^8 per half level), plus the weight and
        // the perturbation rounded to steps: exact int32
        const int32_t Y = (2 * (int32_t)h + 1) * (1 << kAccBits);
        const int32_t Qs = __float2int_rn(__fmul_rn(q, A.acc_R));
        return (xsign ? -Y : Y) + A.acc_W * S + Qs;
    }
}
template <int PREC>
__device__ __forceinline__ bool below(typename Metric<PREC>::T e, uint32_t th_bits) {
    if constexpr (PREC == kFP32 || PREC == kFP16) return e < __uint_as_float(th_bits);
    else return e < (int32_t)th_bits;
}

// Margin byte of a symbol of degree deg with decision sign xsign (see "Lazy evaluation"): a NaN
// takes the low end, where every output is evaluated.
template <int PREC>
__device__ __forceinline__ uint32_t margin_byte(typename Held<PREC>::T h, uint32_t xsign, int deg, const Job& A) {
    float v;
    if constexpr (PREC == kFP32) v = h;
    else if constexpr (PREC == kFP16) v = __half2float(h);
    else v = (float)((2 * (int32_t)h + 1) * (PREC == kFIXACC ? (1 << kAccBits) : 1)) * A.pf_unit;
    v = __uint_as_float(__float_as_uint(v) ^ xsign);
    const float b = __fmaf_rn(v, A.pf_inv, __fmaf_rn(A.pf_w, (float)deg, A.pf_bias));
    return (uint32_t)__float2int_rd(fminf(fmaxf(b, A.pf_lo), A.pf_hi));
}

// Cutoff of margin byte b: no output above it can flip a symbol whose margin is b - kMargin0 steps
// or more.  The relative error of erfcf and of the deviates is covered by the added terms.
__device__ __forceinline__ uint32_t margin_cutoff(int b, const Job& A) {
    if (b <= kMargin0) return 0xFFFFFFFFu;
    const float a = (float)(b - kMargin0) * A.pf_rho - 1e-3f;      // in units of `scale`
    const float p = A.uniform ? 0.5f * (1.0f - a) : 0.5f * erfcf(a * 0.70710678f);
    const float c = p * 4294967296.0f * 1.0001f + 2.0f;
    return a <= 0.0f || c >= 4294967040.0f ? 0xFFFFFFFFu : (c > 0.0f ? (uint32_t)c : 0u);
}

// Objective trace (Sec. III-B objective f(x) = sum_k x_k y_k + sum_i s_i): for the live slots whose
// frame id is below A.trace_frames, records at this syndrome test t the number of unsatisfied
// checks U(t) and C(t) = sum_k rint(x_k(t) y~_k 2^32) (each term exact in double; integer sums are
// independent of their order).  CTA-wide; every thread calls it with the same `live`.
template <int PREC>
__device__ __forceinline__ void trace_round(const Job& A, const SmemLayout& L, const uint16_t* chk_cols,
                                         uint32_t live, int round) {
    extern __shared__ __align__(16) unsigned char smem[];
    const long long* lane_frame = reinterpret_cast<const long long*>(smem + L.off_frame);
    const int32_t* lane_start = reinterpret_cast<const int32_t*>(smem + L.off_start);
    const uint32_t* xw = reinterpret_cast<const uint32_t*>(smem + L.off_xw);
    unsigned long long* tr_c = reinterpret_cast<unsigned long long*>(smem + L.off_trace);
    int32_t* tr_u = reinterpret_cast<int32_t*>(smem + L.off_trace + kSlots * 8);
    const int tid = threadIdx.x, lane = tid & 31;
    const bool mine = ((live >> lane) & 1u) && lane_frame[lane] >= 0 && lane_frame[lane] < A.trace_frames;
    const uint32_t tmask = __ballot_sync(0xFFFFFFFFu, mine);   // the same in every warp
    if (tmask == 0u) return;
    if (tid < kSlots) {
        tr_c[tid] = 0ull;
        tr_u[tid] = 0;
    }
    __syncthreads();
    const int n = A.n, m = A.m;
    // U(t): the syndrome words recomputed from the decision words
    for (int base = 0; base < m; base += blockDim.x) {
        const int i = base + tid;
        uint32_t s = 0u;
        if (i < m)
            for (int j = 0; j < A.dc_max; ++j) s ^= xw[chk_cols[chk_index(j, i, m)]];
        for (uint32_t r = tmask; r; r &= r - 1u) {
            const int f = __ffs(r) - 1;
            const int c = __popc(__ballot_sync(0xFFFFFFFFu, (s >> f) & 1u));
            if (lane == 0 && c) atomicAdd(tr_u + f, c);
        }
    }
    // C(t): sum over symbols of the signed held sample, scaled by 2^32 and rounded
    for (int base = 0; base < n; base += blockDim.x) {
        const int k = base + tid;
        for (uint32_t r = tmask; r; r &= r - 1u) {
            const int f = __ffs(r) - 1;
            long long term = 0;
            if (k < n) {
                const typename Held<PREC>::T h = hold<PREC>(read_sample(A, lane_frame[f], k), A);
                double v;
                if constexpr (PREC == kFP32) {
                    v = (double)h;
                } else if constexpr (PREC == kFP16) {
                    v = (double)__half2float(h);
                } else {
                    v = (double)(2 * (int32_t)h + 1) * A.trace_yunit;
                }
                if ((xw[k] >> f) & 1u) v = -v;
                term = __double2ll_rn(v * 4294967296.0);
            }
#pragma unroll
            for (int o = 16; o; o >>= 1) term += __shfl_xor_sync(0xFFFFFFFFu, term, o);
            if (lane == 0 && term) atomicAdd(tr_c + f, (unsigned long long)term);
        }
    }
    __syncthreads();
    if (tid < kSlots && ((tmask >> tid) & 1u)) {
        const long long fr = lane_frame[tid];
        const size_t at = (size_t)fr * (size_t)(A.t_max + 1) + (size_t)(round - lane_start[tid]);
        A.trace_u[at] = tr_u[tid];
        A.trace_c[at] = (long long)tr_c[tid];
    }
    __syncthreads();
}

// The four held samples of one slot in a group (16, 8 or 4 bytes, aligned).
__device__ __forceinline__ void load_held4(const float* p, float v[4]) {
    const float4 a = *reinterpret_cast<const float4*>(p);
    v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
}
__device__ __forceinline__ void load_held4(const __half* p, __half v[4]) {
    const uint2 a = *reinterpret_cast<const uint2*>(p);
    v[0] = __ushort_as_half((unsigned short)(a.x & 0xFFFFu));
    v[1] = __ushort_as_half((unsigned short)(a.x >> 16));
    v[2] = __ushort_as_half((unsigned short)(a.y & 0xFFFFu));
    v[3] = __ushort_as_half((unsigned short)(a.y >> 16));
}
__device__ __forceinline__ void load_held4(const int8_t* p, int8_t v[4]) {
    const uint32_t a = *reinterpret_cast<const uint32_t*>(p);
    v[0] = (int8_t)(a & 0xFFu); v[1] = (int8_t)((a >> 8) & 0xFFu);
    v[2] = (int8_t)((a >> 16) & 0xFFu); v[3] = (int8_t)(a >> 24);
}

// State word of a symbol after a flip at the slot's iteration t: the flip count, and the window
// count, which takes the new decision for x(t + 1) .. x(T).
template <bool ADAPT, bool SMOOTH>
__device__ __forceinline__ uint32_t flipped_state(uint32_t s0, bool was_neg, int t, int t_max, int t_smooth) {
    uint32_t s1 = s0 + (ADAPT ? 1u : 0u);
    if constexpr (SMOOTH) {
        const uint32_t rem = (uint32_t)(t_max - max(t + 1, t_smooth) + 1) << kCShift;
        s1 = was_neg ? s1 - rem : s1 + rem;
    }
    return s1;
}

// Phase A' (narrow): two threads per group, each for 16 slots: the four symbols' check words added in
// 2-bit lanes three at a time, widened to nibbles (even and odd slots), and the bytes of the four
// symbols gathered into the words that phase C reads.  unit(i, e, d): the (e + d)-th checks of the
// group's symbols, for task i.
template <class Unit>
__device__ __forceinline__ void count_groups(uint4* cnt, const uint32_t* sw, int groups, int dv_max, Unit unit) {
    for (int i = threadIdx.x; i < 2 * groups; i += blockDim.x) {
        const int gl = i >> 1, h = i & 1;
        uint32_t ev[4] = {0u, 0u, 0u, 0u}, od[4] = {0u, 0u, 0u, 0u};
        for (int e = 0; e < dv_max; e += 3) {
            uint32_t a[4] = {0u, 0u, 0u, 0u};
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                if (e + d >= dv_max) break;
                const uint2 c = unit(i, e, d);
                a[0] += sw[2 * (c.x & 0xFFFFu) + h];
                a[1] += sw[2 * (c.x >> 16) + h];
                a[2] += sw[2 * (c.y & 0xFFFFu) + h];
                a[3] += sw[2 * (c.y >> 16) + h];
            }
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                ev[j] += a[j] & 0x33333333u;
                od[j] += (a[j] >> 2) & 0x33333333u;
            }
        }
        auto bytes = [](const uint32_t w[4]) {      // word b: byte b of w[0..3]
            const uint32_t t0 = __byte_perm(w[0], w[1], 0x5140), t1 = __byte_perm(w[0], w[1], 0x7362);
            const uint32_t u0 = __byte_perm(w[2], w[3], 0x5140), u1 = __byte_perm(w[2], w[3], 0x7362);
            return make_uint4(__byte_perm(t0, u0, 0x5410), __byte_perm(t0, u0, 0x7632),
                              __byte_perm(t1, u1, 0x5410), __byte_perm(t1, u1, 0x7632));
        };
        cnt[4 * gl + 2 * h] = bytes(ev);
        cnt[4 * gl + 2 * h + 1] = bytes(od);
    }
}

// Philox round keys as PhiloxLane takes them.
struct PhiloxKeys {
    uint32_t rk0[10], rk1[10];
};

// Iterations with every E_k formed (narrow codes outside clusters, adaptive variants, no trace), lane =
// slot, for a CTA of more than 16 live slots of whose outputs so many are at or below their cutoffs
// that the exact form of those one by one costs more.  Takes over after phase C of iteration `round`,
// in which tally[0] outputs were evaluated; runs phases A, A' and C until a slot finishes or the flips
// say that few outputs would be evaluated, and returns the iteration whose phase A is next.  The slots'
// held samples take the place of their margins in the scratch, and at the end the margins theirs.  A
// function of its own, so that the lazy loop's registers and code are what they are without it.
// 20000 frames, T = 300, all evaluated one by one before this, the former dense form in brackets: (3,6)
// code of 1008 symbols at 0 dB 29.3 -> 18.2 ms (17.2), 1.0 dB 26.4 -> 17.5 (17.2), 2.0 dB 20.0 -> 15.9
// (16.4), 2.5 dB 9.4 (11.9); (6,32) code of 2048 at 2.0 dB 37.5 -> 32.7 (36.8), 3.0 dB 32.1 -> 30.4 (36.8).
template <bool ADAPT, bool SMOOTH, bool ST_SMEM, int PREC, bool CHAIN>
__device__ __noinline__ int full_rounds(const Job& A, const Job* jl, const int8_t* slot_e, int off_icdf, int off_cnt,
                                        int off_xw, int off_sw, int off_thr, int off_st, const uint16_t* chk_cols, const uint16_t* sym_chks, const uint8_t* sym_deg,
                                        int sym_groups, typename Held<PREC>::T* ys, uint16_t* st_cta, uint32_t th0, int round) {
    extern __shared__ __align__(16) unsigned char smem[];
    constexpr bool kState = ADAPT || SMOOTH;
    // (the offsets ahead of the single-bit minima are the same in every narrow layout)
    const SmemLayout L = smem_layout(4, 1, 0, 1, 1, false, false, 0, -1, 0);
    const int n = A.n, m = A.m, T = A.t_max, t_smooth = A.t_smooth, dv_max = A.dv_max, dc8 = (A.dc_max + 7) >> 3;
    const int groups = (n + 3) >> 2;
    const long long* lane_frame = reinterpret_cast<const long long*>(smem + L.off_frame);
    uint32_t* ctl = reinterpret_cast<uint32_t*>(smem + L.off_ctl);
    uint32_t* tally = reinterpret_cast<uint32_t*>(smem + L.off_best);
    const uint4* keys = reinterpret_cast<const uint4*>(tally + 4);
    const float4* icdf = reinterpret_cast<const float4*>(smem + off_icdf);
    uint32_t* xw = reinterpret_cast<uint32_t*>(smem + off_xw);
    uint4* xw4 = reinterpret_cast<uint4*>(xw);
    uint32_t* sw = reinterpret_cast<uint32_t*>(smem + off_sw);
    uint4* cnt = reinterpret_cast<uint4*>(smem + off_cnt);
    const uint32_t* thr = reinterpret_cast<const uint32_t*>(smem + off_thr);
    uint16_t* st = ST_SMEM ? reinterpret_cast<uint16_t*>(smem + off_st) : st_cta;
    const uint32_t* deg4 = reinterpret_cast<const uint32_t*>(sym_deg);
    const uint2* units = reinterpret_cast<const uint2*>(sym_chks);
    const int tid = threadIdx.x, lane = tid & 31, nwarps = blockDim.x >> 5, warp = __shfl_sync(0xFFFFFFFFu, tid >> 5, 0);
    const uint32_t live = ctl[2];
    const bool act = (live >> lane) & 1u;
    auto job_of = [&](int f) -> const Job& { return CHAIN ? jl[slot_e[f]] : A; };
    const float scale = job_of(lane).scale;
    const uint64_t frame = job_of(lane).frame_offset + (uint64_t)(act ? lane_frame[lane] : 0);
    const int start = reinterpret_cast<const int32_t*>(smem + L.off_start)[lane];
    const uint32_t* cntw = reinterpret_cast<const uint32_t*>(cnt) + cnt_word(lane);
    const int csh = cnt_shift(lane);
    const bool uniform = A.uniform != 0;
    const MetricConsts M = {A.w, A.fix_R, A.fix_kmax, A.fix_W, A.acc_R, A.acc_W};
    const int seen = (int)tally[0], most = groups * kFullMarks;

    // the slots' held samples
    for (int k = tid; k < n; k += blockDim.x)
        for (uint32_t r = live; r; r &= r - 1u) {
            const int f = __ffs(r) - 1;
            const Job& Jf = job_of(f);
            ys[gidx(k, f)] = hold<PREC>(read_sample(Jf, lane_frame[f], k), Jf);
        }
    if (tid == 0) tally[1] = tally[2] = 0u;
    __syncthreads();

    uint32_t fin = 0u;
    int least = -1;                     // flips below which it ends (-1: none counted yet)
    for (;;) {
        ++round;
        // ---- A. syndromes (two threads XOR half of a check each) and the vote ----
        uint32_t acc = 0u;
        if (tid == 0) ctl[(round + 1) & 1] = 0u;
        const int h = tid & 1;
        const uint2* cols = reinterpret_cast<const uint2*>(chk_cols);
        for (int base = 0; base < m; base += blockDim.x >> 1) {
            const int i = base + (tid >> 1);
            uint32_t s = 0u;
            if (i < m) {
#pragma unroll 2
                for (int v = 0; v < dc8; ++v) {
                    const uint2 c = cols[2 * (v * m + i) + h];
                    s ^= xw[c.x & 0xFFFFu] ^ xw[c.x >> 16];
                    s ^= xw[c.y & 0xFFFFu] ^ xw[c.y >> 16];
                }
            }
            s ^= __shfl_xor_sync(0xFFFFFFFFu, s, 1);
            if (i < m) sw[2 * i + h] = spread_pairs((s >> (16 * h)) & 0xFFFFu);
            acc |= s;
        }
        acc = __reduce_or_sync(0xFFFFFFFFu, acc);
        if (lane == 0 && acc) atomicOr(ctl + (round & 1), acc);
        __syncthreads();
        const int t = act ? round - start : 0;
        fin = live & (~ctl[round & 1] | __ballot_sync(0xFFFFFFFFu, act && t >= T));
        if (fin) break;
        // (every thread has read the flips of the last iteration, whose word this is)
        if (tid == 0) tally[1 + ((round + 1) & 1)] = 0u;
        // ---- A'. counts of unsatisfied checks ----
        count_groups(cnt, sw, groups, dv_max, [&](int i, int e, int d) { return units[(size_t)(e + d) * sym_groups + (i >> 1)]; });
        __syncthreads();
        // ---- C. Step 2 and Step 3b for every symbol of every live slot, two groups at a time ----
        unsigned flipped = 0;
        PhiloxKeys G;
        {
            const uint4 k0 = keys[0];
            G.rk0[0] = k0.x; G.rk1[0] = k0.y; G.rk0[1] = k0.z; G.rk1[1] = k0.w;
        }
        const PhiloxLane ph(frame, (uint32_t)t, G);
        for (int g0 = 2 * warp; g0 < groups; g0 += 2 * nwarps) {
            const bool two = g0 + 1 < groups;
            const int gs[2] = {g0, two ? g0 + 1 : g0};      // (a single last group twice, once without effect)
            typename Held<PREC>::T yv[2][4];
            [[maybe_unused]] uint2 sv[2];
            uint32_t s4[2], rnd[2][4];
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const int at = (gs[u] * kSlots + lane) * 4;         // this lane's entries in the group layout
                load_held4(ys + at, yv[u]);
                if constexpr (kState) sv[u] = *reinterpret_cast<const uint2*>(st + at);
                // S_k + 64, a byte each
                s4[u] = deg4[gs[u]] + 0x40404040u - 2u * ((cntw[16 * gs[u]] >> csh) & 0x0F0F0F0Fu);
            }
#pragma unroll
            for (int r = 0; r < 5; ++r) {
                const uint4 q = keys[r];
                G.rk0[2 * r] = q.x; G.rk1[2 * r] = q.y; G.rk0[2 * r + 1] = q.z; G.rk1[2 * r + 1] = q.w;
            }
#pragma unroll
            for (int u = 0; u < 2; ++u) ph.group((uint32_t)gs[u], G, rnd[u]);
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const int at = (gs[u] * kSlots + lane) * 4;
                const int have = n - 4 * gs[u];     // (the missing symbols of a partial last group keep their zeros)
                const uint4 x4 = xw4[gs[u]];
                uint32_t fmv[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const uint32_t word = j == 0 ? x4.x : j == 1 ? x4.y : j == 2 ? x4.z : x4.w;
                    const uint32_t xsign = (word << (31 - lane)) & 0x80000000u;
                    const float z = uniform ? uniform_dev(rnd[u][j]) : gauss_icdf(rnd[u][j], icdf);
                    typename Metric<PREC>::T S;
                    // (a byte in the mantissa of 2^23: no conversion instruction)
                    if constexpr (PREC == kFP32 || PREC == kFP16) S = __uint_as_float(__byte_perm(s4[u], 0x4B000000u, 0x7540 + j)) - 8388672.0f;
                    else S = (int)((s4[u] >> (8 * j)) & 0xFFu) - 64;
                    const auto E = metric<PREC>(yv[u][j], xsign, S, __fmul_rn(scale, z), M);
                    [[maybe_unused]] uint32_t s0 = 0u;
                    if constexpr (kState) s0 = j < 2 ? (sv[u].x >> (16 * j)) & 0xFFFFu : (sv[u].y >> (16 * (j - 2))) & 0xFFFFu;
                    const uint32_t th = ADAPT ? thr[(t - (int)(s0 & kUMask)) & kUMask] : th0;
                    const bool flip = below<PREC>(E, th) && act && (u == 0 || two) && (j == 0 || j < have);
                    flipped += flip ? 1u : 0u;
                    if constexpr (kState) {
                        if (flip) st[at + j] = (uint16_t)flipped_state<ADAPT, SMOOTH>(s0, xsign != 0u, t, T, t_smooth);
                    }
                    fmv[j] = __ballot_sync(0xFFFFFFFFu, flip);
                }
                if (lane == 0 && (u == 0 || two))
                    xw4[gs[u]] = make_uint4(x4.x ^ fmv[0], x4.y ^ fmv[1], x4.z ^ fmv[2], x4.w ^ fmv[3]);
            }
        }
        flipped = __reduce_add_sync(0xFFFFFFFFu, flipped);
        if (lane == 0 && flipped) atomicAdd(tally + 1 + (round & 1), flipped);
        __syncthreads();
        // (the flips of the first iteration stand for the outputs evaluated in the one before)
        const int now = (int)tally[1 + (round & 1)];
        if (least < 0) least = (int)(7ll * now * most / (8ll * seen));
        if (now < least) {
            ++round;
            break;
        }
    }
    // ---- the margins of the slots that go on, and of the missing symbols of a partial last group ----
    uint8_t* yb = reinterpret_cast<uint8_t*>(ys);
    __syncthreads();
    if (tid < 2) ctl[tid] = ctl[6 + tid] = 0u;
    for (int k = tid; k < pad4(n); k += blockDim.x) {
        const uint32_t word = k < n ? xw[k] : 0u;
        if (k >= n)
            for (int f = 0; f < kSlots; ++f) yb[gidx(k, f)] = (uint8_t)(int)A.pf_hi;
        else
            for (uint32_t r = live & ~fin; r; r &= r - 1u) {
                const int f = __ffs(r) - 1;
                const Job& Jf = job_of(f);
                yb[gidx(k, f)] = (uint8_t)margin_byte<PREC>(hold<PREC>(read_sample(Jf, lane_frame[f], k), Jf),
                                                            ((word >> f) & 1u) << 31, sym_deg[k], Jf);
            }
    }
    __syncthreads();
    return round;
}

// The slot loop for one job (rows a0-a8 of the method): CTA-wide, returns when the job
// has no unclaimed frame left and every slot of this CTA is idle.  `A` is the job (kernel
// parameters or a shared-memory copy), `thr_src` its thresholds, `L` the shared-memory
// layout of the launch, `ys`/`st_cta` this CTA's slot scratch.
//
// Thread 0 of a CTA whose slots chain serving jobs: gives the slots in `want` new frames,
// claimed from the current entry and, when its job has none left, from other published jobs
// with the same chain key, which ch.next copies into a free entry (one that no slot of `busy`
// or of those just filled refers to).  Sets lane_frame (frame index within its job; -1 for a
// slot left empty), lane_start = start and ch.slot_e for the filled slots; returns them, and
// adds the entries filled to *loaded.
template <class Next>
__device__ uint32_t fill_chained(ChainCtx<Next>& ch, unsigned long long key, uint32_t want, uint32_t busy,
                                 int start, long long* lane_frame, int32_t* lane_start, uint32_t* loaded) {
    uint32_t fresh = 0;
    for (int step = 0; step <= kChain; ++step) {
        const uint32_t left = want & ~fresh;
        if (!left) break;
        const Job& E = ch.jl[*ch.cur_e];
        const int k = __popc(left);
        unsigned long long base = 0;
        if (claim_frames(E, (unsigned)k, &base)) {
            for (int j = 0; j < k; ++j) {
                const int f = nth_set_bit(left, j);
                const unsigned long long fid = base + j;
                if (fid < (unsigned long long)E.n_frames) {
                    lane_frame[f] = (long long)fid;
                    lane_start[f] = start;
                    ch.slot_e[f] = (int8_t)*ch.cur_e;
                    fresh |= 1u << f;
                }
            }
        }
        if (!(want & ~fresh) || key == 0ull) break;
        // the current job has no frames left: another with the same key, into a free entry
        const uint32_t held = busy | fresh;
        int e2 = -1;
        for (int e = 0; e < ch.entries && e2 < 0; ++e) {
            if (e == *ch.cur_e) continue;
            bool used = false;
            for (uint32_t r = held; r; r &= r - 1) used |= ch.slot_e[__ffs(r) - 1] == e;
            if (!used) e2 = e;
        }
        if (e2 < 0 || !ch.next(key, ch.jl[e2])) break;
        *loaded |= 1u << e2;            // its cutoff table is made at the refill
        *ch.cur_e = e2;
    }
    for (uint32_t r = want & ~fresh; r; r &= r - 1) lane_frame[__ffs(r) - 1] = -1;
    return fresh;
}

// Cluster split (CL, S.size > 1): the S.size CTAs of a thread-block cluster decode the same
// 32 slots, each the symbols [S.k_lo, S.k_hi) (samples, state, counts and M(k) rows of those
// only), with a full copy of the decision words in every CTA: each computes all syndromes (so
// the stop vote is the same everywhere), writes the decision words it changes into every
// copy through distributed shared memory, and rank 0 claims frames for the cluster and
// writes the slot table into every CTA.  Cluster barriers separate the phases; every CTA
// takes the same branches (they depend only on the vote and the slot table), so all of them
// reach every barrier.
//
// Chaining (CHAIN, serving): A is ch.jl[0]; when A has no unclaimed frame left, free slots take
// frames of other published jobs with A's chain key (fill_chained), so the CTA keeps its slots
// busy across requests instead of waiting for A's slowest frame; the loop returns when no such
// job has frames left and every slot is idle.
template <bool ADAPT, bool SMOOTH, bool ST_SMEM, bool WIDE, int PREC, bool CL = false, bool CHAIN = false,
          class Next = NoNext>
__device__ __forceinline__ void decode_job(const Job& A, const uint32_t* thr_src, const GenConsts& G,
                                           const SmemLayout& L, int tables,
                                           typename Held<PREC>::T* ys, uint16_t* st_cta,
                                           Split S = Split{0, 1, 0, 0},
                                           ChainCtx<Next> ch = ChainCtx<Next>{nullptr, nullptr, nullptr, Next{}, 0}) {
    static_assert(!(CL && CHAIN), "chained jobs are not split over clusters");
    constexpr bool kState = ADAPT || SMOOTH;
    // the job whose frame slot f holds (per-request fields: samples, sigma, frame offset,
    // outputs, counters); every other field is the same for all chained jobs
    auto job_of = [&](int f) -> const Job& {
        if constexpr (CHAIN) return ch.jl[ch.slot_e[f]];
        return A;
    };
    using HeldT = typename Held<PREC>::T;
    extern __shared__ __align__(16) unsigned char smem[];
    const int n = A.n, m = A.m, T = A.t_max, dv_max = A.dv_max, dc_max = A.dc_max;
    const bool split = CL && S.size > 1;
    const int k_lo = split ? S.k_lo : 0, k_hi = split ? S.k_hi : n;   // this CTA's symbols
    const int nl = k_hi - k_lo;
    // barrier over the CTAs that share the slots (the cluster when split, else this CTA)
    auto group_sync = [&]() {
        if constexpr (CL) {
            if (split) {
                cooperative_groups::this_cluster().sync();
                return;
            }
        }
        __syncthreads();
    };
    // the same shared-memory word in another CTA of the cluster
    auto peer = [&](auto* p, int r) { return cooperative_groups::this_cluster().map_shared_rank(p, r); };
    long long* lane_frame = reinterpret_cast<long long*>(smem + L.off_frame);
    int32_t* lane_start = reinterpret_cast<int32_t*>(smem + L.off_start);
    uint32_t* ctl = reinterpret_cast<uint32_t*>(smem + L.off_ctl);
    int32_t* unsat_n = reinterpret_cast<int32_t*>(smem + L.off_unsat);
    uint32_t* flips = reinterpret_cast<uint32_t*>(smem + L.off_flips);
    uint4* cnt = reinterpret_cast<uint4*>(smem + L.off_cnt);
    uint32_t* xw = reinterpret_cast<uint32_t*>(smem + L.off_xw);
    uint32_t* sw = reinterpret_cast<uint32_t*>(smem + L.off_sw);
    unsigned long long* best = reinterpret_cast<unsigned long long*>(smem + L.off_best);
    float4* icdf = reinterpret_cast<float4*>(smem + L.off_icdf);
    uint32_t* cut = reinterpret_cast<uint32_t*>(smem + L.off_cut);
    float* tau = reinterpret_cast<float*>(smem + L.off_tau);
    const bool single = !ADAPT && A.single;
    // wide: every symbol evaluated, with its held sample in `ys`; else margin bytes there
    constexpr bool dense = WIDE;
    // syndromes and counts kept between iterations and moved by the flips when these are few
    const bool keep = !WIDE && !split;
    // D: lanes per check of a flip, 1 / dv_max (16 fraction bits), and the flips up to which it is
    // used: their checks fit the queues' memory, and their shared atomics (about 2 lanes per cycle,
    // d_v d_c a flip) cost less than forming all syndromes and counts: 32 flips for the (6,32) code of
    // 2048 symbols, 63 for the (3,6) code of 1008 (16 to 64 measured alike, 128 slower by 3 to 40 %)
    const int sg_log = dc_max > 16 ? 5 : (dc_max > 1 ? 32 - __clz(dc_max - 1) : 0);
    const int dv_inv = (65536 + dv_max - 1) / dv_max;
    const int few = min(min(kFlips, 32 * kQueue / dv_max), max(16, n / (2 << sg_log)));
    const bool record = keep && (tables & kTight) == 0;
    uint8_t* yb = reinterpret_cast<uint8_t*>(ys);
    uint32_t* thr = ADAPT ? reinterpret_cast<uint32_t*>(smem + L.off_thr) : nullptr;
    uint16_t* st = nullptr;
    if constexpr (kState) {
        st = ST_SMEM ? reinterpret_cast<uint16_t*>(smem + L.off_st) : st_cta;
    }
    const int tid = threadIdx.x, lane = tid & 31, nwarps = blockDim.x >> 5, nw_log = 31 - __clz(nwarps);
    const int warp = __shfl_sync(0xFFFFFFFFu, tid >> 5, 0);      // uniform, and known to be
    // adjacency tables: only phases A and A' read them, so a generic pointer to
    // shared or global memory serves both placements
    const uint16_t* chk_cols = A.chk_cols;
    const uint16_t* sym_chks = A.sym_chks;
    const uint8_t* sym_deg = A.sym_deg;
    if (tables & kTabChk) {
        uint16_t* c = reinterpret_cast<uint16_t*>(smem + L.off_chk);
        const uint32_t* src = reinterpret_cast<const uint32_t*>(A.chk_cols);
        for (int i = tid; i < chk_entries(m, dc_max) / 2; i += blockDim.x) reinterpret_cast<uint32_t*>(c)[i] = src[i];
        chk_cols = c;
    }
    int sym_base = 0;           // first symbol that sym_deg (and a shared-memory M(k)) begins with
    // M(k) in 8-byte units, one per (j, group of four symbols): the j-th checks of the four
    int sym_groups = pad4(n) >> 2, sym_g0 = k_lo >> 2;     // units per j; unit of this CTA's first group
    if (tables & kTabSym) {
        uint16_t* s = reinterpret_cast<uint16_t*>(smem + L.off_sym);
        uint8_t* d = reinterpret_cast<uint8_t*>(s + pad4(nl) * dv_max);
        const int gl = pad4(nl) >> 2;
        for (int i = tid; i < gl * dv_max; i += blockDim.x)
            reinterpret_cast<uint2*>(s)[i] = reinterpret_cast<const uint2*>(A.sym_chks)[(size_t)(i / gl) * sym_groups + sym_g0 + i % gl];
        for (int i = tid; i < nl; i += blockDim.x) d[i] = A.sym_deg[k_lo + i];
        sym_chks = s;
        sym_deg = d;
        sym_base = k_lo;
        sym_groups = gl;
        sym_g0 = 0;
    }

    // ---- the first 32 frames, then the set-up: generator table, zeroed state, sentinels,
    // thresholds.  Unsplit, the claim comes first, so that a CTA that finds every frame taken
    // (several CTAs pick a job at once) returns without the set-up. ----
    auto claim_first = [&]() {          // thread 0 (rank 0 when split): slot table and live mask
        uint32_t live = 0;
        for (int c = 0; c < 8; ++c) ctl[c] = 0u;
        if constexpr (CHAIN) {
            *ch.cur_e = 0;
            for (int f = 0; f < kSlots; ++f) ch.slot_e[f] = 0;     // every slot names a loaded entry
            live = fill_chained(ch, A.chain_key, 0xFFFFFFFFu, 0u, 0, lane_frame, lane_start, ctl + 4);
        } else {
            unsigned long long base = 0;
            const unsigned first = busy_slots(A);
            const bool got = claim_frames(A, first, &base);
            for (int f = 0; f < kSlots; ++f) {
                const unsigned long long fid = base + f;
                lane_start[f] = 0;
                if (got && f < (int)first && fid < (unsigned long long)A.n_frames) {
                    lane_frame[f] = (long long)fid;
                    live |= 1u << f;
                } else {
                    lane_frame[f] = -1;
                }
            }
        }
        ctl[2] = live;
        ctl[3] = live;
        if (!CHAIN && A.in_flight != nullptr && live) {
            ctl[4] = (uint32_t)__popc(live);
            atomicAdd(A.in_flight, ctl[4]);
        }
        return live;
    };
    if (!split) {
        if (tid == 0) claim_first();
        __syncthreads();
        if (ctl[2] == 0u) return;
    }
    for (int i = tid; i < 256; i += blockDim.x) icdf[i] = G.icdf[i];
    for (int k = tid; k < pad4(n + 1); k += blockDim.x) xw[k] = 0u;
    for (int i = tid; i < (m + 1) * (WIDE ? 1 : 2); i += blockDim.x) sw[i] = 0u;
    // (an unsplit chaining CTA makes entry 0's table here, the others' when they are loaded)
    if constexpr (!WIDE)
        for (int i = tid; i < 256; i += blockDim.x) cut[i] = margin_cutoff(i, A);
    // the missing symbols of a partial last group: margins that nothing undercuts
    if (!dense)
        for (int e = nl * kSlots + tid; e < pad4(nl) * kSlots; e += blockDim.x)
            yb[gidx(e / kSlots, e % kSlots)] = (uint8_t)(int)A.pf_hi;
    // a serving job's thresholds and samples were copied in while the kernel runs: read them
    // past L1, which may still hold lines of an earlier request at the same addresses
    if constexpr (ADAPT)
        for (int u = tid; u <= T; u += blockDim.x) thr[u] = A.gen ? __ldcg(thr_src + u) : thr_src[u];
    // threshold of the non-adaptive variants; chained jobs read it once here, since the first
    // job's memory is returned when that job completes
    const uint32_t th0_once = CHAIN ? __ldcg(thr_src) : 0u;
    // not single-bit: the outputs evaluated in an iteration, the flips of one of full_rounds (two, by
    // parity), and at 16 bytes the generator's round keys for it
    uint32_t* tally = reinterpret_cast<uint32_t*>(best);
    if (tid < (CHAIN ? 1 : 2) * kSlots)
        best[tid] = single ? ~0ull : tid >= 2 && tid < 12 ? (unsigned long long)G.rk1[tid - 2] << 32 | G.rk0[tid - 2] : 0ull;
    if (split) {
        group_sync();        // every copy cleared before rank 0 writes the slot table
        if (tid == 0 && S.rank == 0) {
            const uint32_t live = claim_first();
            if constexpr (CL) {
                for (int r = 0; r < S.size; ++r) {
                    if (r == S.rank) continue;
                    long long* pf = peer(lane_frame, r);
                    int32_t* ps = peer(lane_start, r);
                    uint32_t* pc = peer(ctl, r);
                    for (int f = 0; f < kSlots; ++f) {
                        pf[f] = lane_frame[f];
                        ps[f] = 0;
                    }
                    for (int c = 0; c < 8; ++c) pc[c] = 0u;
                    pc[2] = live;
                    pc[3] = live;
                }
            }
        }
    }
    group_sync();

    int round = 0;   // flip phases executed by this CTA; slot f is at t = round - lane_start[f]
    int pass_id = 0;
    bool refill = true;
    bool anew = true;   // syndromes and counts formed from the decisions (else kept, D)
    for (;;) {
        if (refill) {
            // ---- load new frames: saturated samples into the slot columns, x(0) = sign(y) ----
            // (four samples in flight per thread)
            const uint32_t fresh = ctl[3];
            if (!dense && single && tid < kSlots && ((fresh >> tid) & 1u)) tau[tid] = A.pf_low + kFirst * job_of(tid).scale;
            if constexpr (CHAIN && !WIDE) {
                for (uint32_t r = ctl[4]; r; r &= r - 1) {
                    const int e = __ffs(r) - 1;
                    for (int i = tid; i < 256; i += blockDim.x) cut[256 * e + i] = margin_cutoff(i, ch.jl[e]);
                }
            }
            for (int k = k_lo + tid; k < k_hi; k += blockDim.x) {
                uint32_t word = xw[k] & ~fresh;
                const int deg = sym_deg[k - sym_base];
                for (uint32_t rest = fresh; rest;) {
                    int fs[4];
                    float v[4];
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        fs[i] = __ffs(rest) - 1;            // -1 when none is left
                        rest &= rest - 1;
                        v[i] = fs[i] >= 0 ? read_sample(job_of(fs[i]), lane_frame[fs[i]], k) : 0.0f;
                    }
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const int f = fs[i];
                        if (f < 0) break;
                        const Job& Jf = job_of(f);
                        const HeldT h = hold<PREC>(v[i], Jf);
                        const bool negative = held_negative<PREC>(h);
                        const int at = gidx(k - k_lo, f);
                        if (dense) ys[at] = h;
                        else yb[at] = (uint8_t)margin_byte<PREC>(h, negative ? 0x80000000u : 0u, deg, Jf);
                        if (negative) word |= 1u << f;
                        // no flips yet; without any, every x(t) of the window is x(0)
                        if constexpr (kState)
                            st[at] = (SMOOTH && negative) ? (uint16_t)((T - A.t_smooth + 1) << kCShift) : 0;
                    }
                }
                xw[k] = word;
                if constexpr (CL) {
                    for (int r = 0; split && r < S.size; ++r)
                        if (r != S.rank) peer(xw, r)[k] = word;
                }
            }
            group_sync();
            if (CHAIN && tid == 0) ctl[4] = 0u;
            refill = false;
            anew = true;
        }

        const uint2* units = reinterpret_cast<const uint2*>(sym_chks) + sym_g0;
        const int groups_l = (nl + 3) >> 2;          // groups of four symbols (the code's last can be partial)
        [[maybe_unused]] uint2 pre[3] = {};
        if (anew) {
            // the first checks of this thread's symbols (phase A'), fetched while the syndromes form
            if constexpr (!WIDE) {
                if (tid < 2 * groups_l) {
#pragma unroll
                    for (int d = 0; d < 3; ++d)
                        if (d < dv_max) pre[d] = units[(size_t)d * sym_groups + (tid >> 1)];
                }
            }
            // ---- A. syndromes (two threads XOR half of a check each) and the vote ----
            uint32_t* unsat = ctl + (pass_id & 1);
            if (tid == 0) ctl[(pass_id + 1) & 1] = 0u;
            if (keep) {
                if (tid < kSlots) unsat_n[tid] = 0;
                __syncthreads();
            }
            uint32_t acc = 0;
            int open = 0;                // unsatisfied checks of slot `lane` seen by this warp
            const int h = tid & 1, dc8 = (dc_max + 7) >> 3;
            const uint2* cols = reinterpret_cast<const uint2*>(chk_cols);
            for (int base = 0; base < m; base += blockDim.x >> 1) {
                const int i = base + (tid >> 1);
                uint32_t s = 0;
                if (i < m) {
#pragma unroll 2
                    for (int v = 0; v < dc8; ++v) {
                        const uint2 c = cols[2 * (v * m + i) + h];
                        s ^= xw[c.x & 0xFFFFu] ^ xw[c.x >> 16];
                        s ^= xw[c.y & 0xFFFFu] ^ xw[c.y >> 16];
                    }
                }
                s ^= __shfl_xor_sync(0xFFFFFFFFu, s, 1);
                if constexpr (WIDE) {
                    if (i < m && h == 0) sw[i] = s;
                } else {
                    // half h of the word, one slot per 2-bit lane (slots 16 h .. 16 h + 15)
                    if (i < m) sw[2 * i + h] = spread_pairs((s >> (16 * h)) & 0xFFFFu);
                }
                if (keep) open += column_count(h ? 0u : s, lane);
                else acc |= s;
            }
            if (keep) {
                if (open) atomicAdd(unsat_n + lane, open);
            } else {
                acc = __reduce_or_sync(0xFFFFFFFFu, acc);
                if (lane == 0 && acc) atomicOr(unsat, acc);
            }
            __syncthreads();
        }
        const uint32_t unsat = keep ? __ballot_sync(0xFFFFFFFFu, unsat_n[lane] != 0) : ctl[pass_id & 1];
        if (anew) ++pass_id;
        uint32_t live = ctl[2];
        if (A.trace_u != nullptr)
            trace_round<PREC>(A, L, chk_cols, live, round);
        const uint32_t conv = live & ~unsat;
        const int my_t = round - lane_start[lane];
        const uint32_t at_T = __ballot_sync(0xFFFFFFFFu, ((live >> lane) & 1u) && my_t >= T);
        const uint32_t fin = conv | (live & at_T);

        if (fin) {
            // ---- B. outputs of finished slots ----
            const int nfin = __popc(fin);
            const int b_lo = k_lo >> 3, nbl = ((k_hi + 7) >> 3) - b_lo;   // this CTA's output bytes
            const int work = nfin * nbl;
            for (int idx = tid; idx < work; idx += blockDim.x) {
                const int j = idx / nbl, b = b_lo + (idx - j * nbl);
                const int f = nth_set_bit(fin, j);
                const bool ok = (conv >> f) & 1u;
                const int tf = round - lane_start[f];
                uint32_t byte = 0;
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                    const int k = 8 * b + q;
                    if (k < n) {
                        uint32_t bit = (xw[k] >> f) & 1u;
                        if constexpr (SMOOTH) {
                            if (!ok) {
                                // X_k = terms - 2 * (#-1 decisions in t_smooth .. T)
                                const int terms = tf - A.t_smooth + 1;
                                const int neg = (int)(st[gidx(k - k_lo, f)] >> kCShift);
                                const int X = terms - 2 * neg;
                                bit = X < 0 ? 1u : (X > 0 ? 0u : bit);
                            }
                        }
                        byte |= bit << q;
                    }
                }
                job_of(f).bits[(size_t)lane_frame[f] * A.nb + b] = (uint8_t)byte;
            }
            if (tid < nfin && (!split || S.rank == 0)) {
                const int f = nth_set_bit(fin, tid);
                const bool ok = (conv >> f) & 1u;
                const long long fr = lane_frame[f];
                const Job& Jf = job_of(f);
                Jf.iters[fr] = ok ? round - lane_start[f] : T;
                Jf.pass[fr] = ok ? 1 : 0;
            }
            if (A.done != nullptr) __threadfence();   // outputs visible before they are counted
            group_sync();           // every CTA is done with the finished slots' table entries
            if (A.done != nullptr && tid == 0 && (!split || S.rank == 0)) {
                if constexpr (CHAIN) {
                    // the finished frames counted in their own jobs
                    for (int e = 0; e < kChain; ++e) {
                        int cnt = 0;
                        for (uint32_t r = fin; r; r &= r - 1)
                            cnt += ch.slot_e[__ffs(r) - 1] == e ? 1 : 0;
                        if (!cnt) continue;
                        const Job& E = ch.jl[e];
                        const unsigned int before = atomicAdd(E.done, (unsigned int)cnt);
                        if ((long long)before + cnt == E.n_frames) {
                            __threadfence_system();
                            *(volatile unsigned int*)E.notify = E.gen;
                        }
                    }
                } else {
                    const unsigned int before = atomicAdd(A.done, (unsigned int)nfin);
                    if ((long long)before + nfin == A.n_frames) {
                        __threadfence_system();
                        *(volatile unsigned int*)A.notify = A.gen;
                    }
                }
            }
            // ---- claim new frames for the finished slots ----
            if (tid == 0 && (!split || S.rank == 0)) {
                uint32_t fresh = 0;
                if constexpr (CHAIN) {
                    // (the finished slots and any that were left empty)
                    fresh = fill_chained(ch, A.chain_key, ~(live & ~fin), live & ~fin, round, lane_frame, lane_start, ctl + 4);
                } else {
                    unsigned long long base = 0;
                    const bool got = claim_frames(A, (unsigned)nfin, &base);
                    for (int j = 0; j < nfin; ++j) {
                        const int f = nth_set_bit(fin, j);
                        const unsigned long long fid = base + j;
                        if (got && fid < (unsigned long long)A.n_frames) {
                            lane_frame[f] = (long long)fid;
                            lane_start[f] = round;
                            fresh |= 1u << f;
                        } else {
                            lane_frame[f] = -1;
                        }
                    }
                }
                ctl[2] = (live & ~fin) | fresh;
                ctl[3] = fresh;
                if constexpr (CL) {
                    for (int r = 0; split && r < S.size; ++r) {
                        if (r == S.rank) continue;
                        long long* pf = peer(lane_frame, r);
                        int32_t* ps = peer(lane_start, r);
                        uint32_t* pc = peer(ctl, r);
                        for (int j = 0; j < nfin; ++j) {
                            const int f = nth_set_bit(fin, j);
                            pf[f] = lane_frame[f];
                            ps[f] = lane_start[f];
                        }
                        pc[2] = ctl[2];
                        pc[3] = ctl[3];
                    }
                }
            }
            group_sync();
            live = ctl[2];
            if (ctl[3]) {
                refill = true;      // new frames need their t = 0 syndrome test first
                continue;
            }
        }
        if (live == 0) break;

        // ---- A'. per symbol and slot, the count of unsatisfied checks in M(k) ----
        uint32_t* n_flips = ctl + 6 + (round & 1);
        if (tid == 0) ctl[6 + ((round + 1) & 1)] = 0u;
        if (!WIDE && !CL && ADAPT && !single && tid == 0 && (round & kFullEvery) == kFullEvery - 1) tally[0] = 0u;
        if (anew) {
        // a CTA of a split job flips decisions in every copy during phase C: none before every
        // CTA has formed its syndromes (the barrier's wait is below, after the counts)
        if constexpr (CL) {
            if (split) cooperative_groups::this_cluster().barrier_arrive();
        }
        if constexpr (!WIDE) {
            count_groups(cnt, sw, groups_l, dv_max, [&](int i, int e, int d) {
                return i == tid && e == 0 ? pre[d] : units[(size_t)(e + d) * sym_groups + (i >> 1)];
            });
        } else {
            for (int k = k_lo + tid; k < k_hi; k += blockDim.x) {
                const int kk = k - k_lo;                      // local index of the symbol
                const uint16_t* row = sym_chks + 4 * (size_t)(sym_g0 + (kk >> 2)) + (k & 3);
                uint32_t b[7] = {0, 0, 0, 0, 0, 0, 0};     // count <= 127: seven slices
                for (int e = 0; e < dv_max; ++e) {
                    uint32_t carry = sw[row[4 * (size_t)e * sym_groups]];
#pragma unroll
                    for (int q = 0; q < 7; ++q) {
                        const uint32_t c = b[q] & carry;
                        b[q] ^= carry;
                        carry = c;
                    }
                }
                cnt[2 * kk] = make_uint4(b[0], b[1], b[2], b[3]);
                cnt[2 * kk + 1] = make_uint4(b[4], b[5], b[6], (uint32_t)sym_deg[k - sym_base]);
            }
        }
        if constexpr (CL) {
            if (split) cooperative_groups::this_cluster().barrier_wait();
        }
        __syncthreads();
        }

        // threshold of the non-adaptive variants
        const uint32_t th0 = CHAIN ? th0_once : (A.gen ? __ldcg(thr_src) : thr_src[0]);
        const int g_lo = k_lo >> 2;              // first group of this CTA's symbols
        const uint32_t* cntw = reinterpret_cast<const uint32_t*>(cnt);
        const bool uniform = A.uniform != 0;

        // A flip of (symbol kl of this CTA, slot f) at the slot's iteration t
        auto flip_at = [&](uint32_t s0, bool was_neg, int t) -> uint32_t {
            return flipped_state<ADAPT, SMOOTH>(s0, was_neg, t, T, A.t_smooth);
        };

        // E_k as an order-preserving key and, from the key, in real units (single-bit variant)
        auto key_of = [](typename Metric<PREC>::T E) -> uint32_t {
            if constexpr (PREC == kFP32 || PREC == kFP16) return order_key(E);
            else return (uint32_t)E ^ 0x80000000u;
        };
        auto value_of = [&](uint32_t key) -> float {
            if constexpr (PREC == kFP32 || PREC == kFP16)
                return __uint_as_float((key & 0x80000000u) ? key ^ 0x80000000u : ~key);
            else return __fmul_rn((float)(int32_t)(key ^ 0x80000000u), A.pf_unit);
        };
        // single-bit variant: least (E key, k) of each slot over this CTA's symbols; when split, in
        // the buffer of this round's parity (the CTAs of the cluster read each other's)
        unsigned long long* bcur = best + (split ? (round & 1) * kSlots : 0);
        uint32_t todo = live;           // single-bit variant: slots whose flip is not decided yet

        // ---- C. Step 2 and Step 3b for every symbol of every live slot ----
        for (int sweep = 1;; ++sweep) {
        if constexpr (!dense) {
            // lanes over (group, slot): several groups at a time when few slots are live
            const int n_live = __popc(todo);
            const int lg = n_live > 1 ? 32 - __clz(n_live - 1) : 0;
            const int li = lane & ((1 << lg) - 1);
            const bool act = li < n_live;
            const int slot = n_live == 32 ? lane : select_bit(todo, act ? li : 0);
            const Job& Jl = job_of(slot);
            const int t = round - lane_start[slot];
            const PhiloxLane ph(Jl.frame_offset + (uint64_t)lane_frame[slot], (uint32_t)t, G);
            uint32_t K = (uint32_t)Jl.pf_K, D = 0u, ebase = 0u;
            [[maybe_unused]] uint32_t shift = 0u;        // single-bit: steps off every margin, down to 0
            if constexpr (ADAPT) {
                const float th = (PREC == kFP32 || PREC == kFP16) ? __uint_as_float(thr[t]) : (float)(int32_t)thr[t];
                const float d = __fmaf_rn(-Jl.pf_d1, th, Jl.pf_d0);
                D = (uint32_t)min((int)fminf(fmaxf(d, 0.0f), 255.0f), Jl.pf_dcap) * 0x01010101u;
            } else if (single) {
                shift = (uint32_t)-__float2int_rd(fminf(fmaxf(__fmaf_rn(-Jl.pf_d1, tau[slot], Jl.pf_d0), -255.0f), 0.0f)) * 0x01010101u;
            }
            if constexpr (CHAIN) ebase = (uint32_t)ch.slot_e[slot];
            const uint32_t csh = (uint32_t)cnt_shift(slot);
            // queue: local group | slot << 16 | outputs at or below their cutoffs << 24
            uint32_t* queue = reinterpret_cast<uint32_t*>(smem + L.off_queue) + warp * kQueue;
            int queued = 0, evaluated = 0;

            // the exact form for one output of one symbol per lane that is `on`: E_k, its flip (or, in the
            // single-bit variant, its claim to be the slot's least)
            auto settle = [&](bool on, int kl, int f, uint32_t out) {
                bool flip = false;
                const int k = k_lo + kl;
                if (on && k < k_hi) {
                    const Job& Jf = job_of(f);
                    const HeldT h = hold<PREC>(read_sample(Jf, lane_frame[f], k), Jf);
                    const int tf = round - lane_start[f];
                    const int deg = sym_deg[k - sym_base];
                    const uint32_t c = (cntw[(kl >> 2) * 16 + cnt_word(f)] >> (8 * (kl & 3) + cnt_shift(f))) & 0xFu;
                    uint32_t* xk = xw + k;
                    const uint32_t xsign = ((*(volatile uint32_t*)xk >> f) & 1u) << 31;
                    const float z = uniform ? uniform_dev(out) : gauss_icdf(out, icdf);
                    const auto E = metric<PREC>(h, xsign, deg - 2 * (int)c, __fmul_rn(Jf.scale, z), A);
                    if (single) {
                        // Step 3a: the slot's least E_k (the lowest k among equal values)
                        const unsigned long long cand = ((unsigned long long)key_of(E) << 32) | (uint32_t)k;
                        if (cand < *(volatile unsigned long long*)(bcur + f)) atomicMin(bcur + f, cand);
                    } else {
                        const int at = gidx(kl, f);
                        [[maybe_unused]] uint32_t s0 = 0u;
                        if constexpr (kState) s0 = st[at];
                        flip = below<PREC>(E, ADAPT ? thr[(tf - (int)(s0 & kUMask)) & kUMask] : th0);
                        if (flip) {
                            atomicXor(xk, 1u << f);
                            if constexpr (CL) {
                                for (int r = 0; split && r < S.size; ++r)
                                    if (r != S.rank) atomicXor(peer(xw, r) + k, 1u << f);
                            }
                            if constexpr (kState) st[at] = (uint16_t)flip_at(s0, xsign != 0u, tf);
                            yb[at] = (uint8_t)margin_byte<PREC>(h, xsign ^ 0x80000000u, deg, Jf);
                        }
                    }
                }
                // recorded while they are few enough to be used (D); the warp takes one lane's reading of
                // the count, since other warps add to it meanwhile
                const uint32_t fl = __ballot_sync(0xFFFFFFFFu, flip);
                if (fl && record && __shfl_sync(0xFFFFFFFFu, *(volatile uint32_t*)n_flips, 0) <= (uint32_t)few) {
                    int at = 0;
                    if (lane == 0) at = (int)atomicAdd(n_flips, (unsigned)__popc(fl));
                    at = __shfl_sync(0xFFFFFFFFu, at, 0) + __popc(fl & ((1u << lane) - 1u));
                    if (flip && at < kFlips) flips[at] = (uint32_t)kl | ((uint32_t)f << 16);
                }
            };
            // the exact form for the first marked output of the last `count` queued groups, one group
            // per lane (its outputs drawn again: four bytes queued instead of twenty, and nothing of
            // the draw kept in the sweep); groups with further marks go back into the queue
            auto evaluate = [&](int count) {
                __syncwarp();
                evaluated += count;
                queued -= count;
                const uint32_t q = lane < count ? queue[queued + lane] : 0u;
                const int f = q ? (int)((q >> 16) & 31u) : slot, j = (__ffs(q >> 24) - 1) & 3, g = (int)(q & 0xFFFFu);
                uint32_t r[4];
                PhiloxLane(job_of(f).frame_offset + (uint64_t)lane_frame[f], (uint32_t)(round - lane_start[f]), G)
                    .group((uint32_t)(g_lo + g), G, r);
                settle(q != 0u, 4 * g + j, f, j & 2 ? (j & 1 ? r[3] : r[2]) : (j & 1 ? r[1] : r[0]));
                uint32_t rest = q & ~(1u << (24 + j));
                if ((rest >> 24) == 0u) rest = 0u;
                const uint32_t back = __ballot_sync(0xFFFFFFFFu, rest != 0u);
                if (rest) queue[queued + __popc(back & ((1u << lane) - 1u))] = rest;
                queued += __popc(back);
                __syncwarp();
            };

            // Steps of one or more groups, a contiguous range of them per warp (the lanes past the code's
            // last group or without a slot compute on what they read and are masked where outputs are
            // queued).  With every lane on a slot of its own (ALL) a step is one group, the strides are
            // constants, the first generator rounds' products of the group uniform, and two steps go
            // together for their independent chains; with fewer slots there are few steps per warp.
            auto run = [&](auto all_tag) {
                constexpr bool ALL = decltype(all_tag)::value;
                constexpr int U = ALL ? 2 : 1;
                const int lgs = ALL ? 5 : lg, stride = 1 << (5 - lgs);
                const int steps = (groups_l + stride - 1) >> (5 - lgs);
                const int each = ((steps + U * nwarps - 1) >> (nw_log + U - 1)) * U;
                const int s_end = min((warp + 1) * each, steps);
                int gl = ((warp * each) << (5 - lgs)) + (ALL ? 0 : lane >> lgs);
                const uint32_t* yp = reinterpret_cast<const uint32_t*>(yb) + (size_t)gl * kSlots + slot;
                const uint32_t* cp = cntw + gl * 16 + cnt_word(slot);
                for (int step = warp * each; step < s_end; step += U) {
                    // the loads before the generator's arithmetic, so that their latency overlaps it
                    uint32_t y4[U], c4[U], r[U][4];
#pragma unroll
                    for (int u = 0; u < U; ++u) {
                        y4[u] = yp[u * stride * kSlots];
                        c4[u] = cp[u * stride * 16];
                    }
#pragma unroll
                    for (int u = 0; u < U; ++u) ph.group((uint32_t)(g_lo + gl + u * stride), G, r[u]);
                    bool low[U][4], any = false;
#pragma unroll
                    for (int u = 0; u < U; ++u) {
                        uint32_t m4 = y4[u] + D - K * ((c4[u] >> csh) & 0x0F0F0F0Fu);
                        if (single) m4 = __vsubus4(m4, shift);
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            low[u][j] = r[u][j] <= cut[__byte_perm(m4, ebase, 0x5540 + j)];
                            any = any || low[u][j];
                        }
                    }
                    if (__any_sync(0xFFFFFFFFu, any)) {
                        uint32_t mark[U];
#pragma unroll
                        for (int u = 0; u < U; ++u) {
                            mark[u] = (low[u][0] ? 1u : 0u) | (low[u][1] ? 2u : 0u) | (low[u][2] ? 4u : 0u) | (low[u][3] ? 8u : 0u);
                            if (!(act && step + u < s_end && gl + u * stride < groups_l)) mark[u] = 0u;
                        }
                        if (ALL || each > 2) {
                            uint32_t b[U];
#pragma unroll
                            for (int u = 0; u < U; ++u) b[u] = __ballot_sync(0xFFFFFFFFu, mark[u] != 0u);
                            const uint32_t lt = (1u << lane) - 1u;
                            const uint32_t what = (uint32_t)gl | ((uint32_t)slot << 16);
                            if (mark[0]) queue[queued + __popc(b[0] & lt)] = what | (mark[0] << 24);
                            queued += __popc(b[0]);
                            while (queued >= 32) evaluate(32);
                            if constexpr (U > 1) {
                                if (mark[U - 1]) queue[queued + __popc(b[U - 1] & lt)] = (what + stride) | (mark[U - 1] << 24);
                                queued += __popc(b[U - 1]);
                                while (queued >= 32) evaluate(32);
                            }
                        } else {
                            // few steps per warp: its own outputs at once, for the shorter way to the barrier
                            uint32_t mk = mark[0];
                            while (__any_sync(0xFFFFFFFFu, mk != 0u)) {
                                const int j = (__ffs(mk) - 1) & 3;
                                settle(mk != 0u, 4 * gl + j, slot, j & 2 ? (j & 1 ? r[0][3] : r[0][2]) : (j & 1 ? r[0][1] : r[0][0]));
                                mk &= mk - 1u;
                            }
                        }
                    }
                    gl += U * stride;
                    yp += U * stride * kSlots;
                    cp += U * stride * 16;
                }
            };
            if (lg == 5) run(std::true_type{});
            else run(std::false_type{});
            while (queued) evaluate(queued < 32 ? queued : 32);
            if (!CL && ADAPT && !single && (round & kFullEvery) == kFullEvery && lane == 0 && evaluated) atomicAdd(tally, (unsigned)evaluated);
        } else {
            // every symbol of every slot, lane = slot (an idle slot's decisions and counters are
            // don't-care: cleared when it takes a frame, never part of an output)
            const bool act = (live >> lane) & 1u;
            const long long fr = lane_frame[lane];
            const Job& Jl = job_of(lane);
            const uint64_t fid = Jl.frame_offset + (uint64_t)(act ? fr : 0);
            const uint32_t flo = (uint32_t)fid, fhi = (uint32_t)(fid >> 32);
            const int t = act ? round - lane_start[lane] : 0;
            const float scale = Jl.scale;
            unsigned long long my_best = ~0ull;      // single-bit variant: (E key << 32) | k
            for (int gl = warp; gl < groups_l; gl += nwarps) {
                const int g = g_lo + gl, k0 = 4 * g;     // group index in the code (Philox counter)
                const int at = (gl * kSlots + lane) * 4;  // this lane's entries in the group layout
                HeldT yv[4];
                load_held4(ys + at, yv);
                [[maybe_unused]] uint32_t sv[4] = {0u, 0u, 0u, 0u};
                if constexpr (kState) {
                    const uint2 s2 = *reinterpret_cast<const uint2*>(st + at);
                    sv[0] = s2.x & 0xFFFFu; sv[1] = s2.x >> 16; sv[2] = s2.y & 0xFFFFu; sv[3] = s2.y >> 16;
                }
                const uint4 x4 = reinterpret_cast<const uint4*>(xw)[g];
                const uint32_t xwv[4] = {x4.x, x4.y, x4.z, x4.w};
                float z[4];
                noise4((uint32_t)g, (uint32_t)t, flo, fhi, G, icdf, uniform, z);
                uint32_t fmv[4] = {0u, 0u, 0u, 0u};          // flip masks of the four symbols
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const int k = k0 + j;
                    if (k >= k_hi) break;
                    const uint4 c = cnt[2 * (k - k_lo)], d = cnt[2 * (k - k_lo) + 1];
                    const int unsat_cnt = (int)(((c.x >> lane) & 1u) | (((c.y >> lane) & 1u) << 1) |
                                                (((c.z >> lane) & 1u) << 2) | (((c.w >> lane) & 1u) << 3) |
                                                (((d.x >> lane) & 1u) << 4) | (((d.y >> lane) & 1u) << 5) |
                                                (((d.z >> lane) & 1u) << 6));
                    const int Sk = (int)d.w - 2 * unsat_cnt;
                    const uint32_t xsign = (xwv[j] << (31 - lane)) & 0x80000000u;
                    const auto E = metric<PREC>(yv[j], xsign, Sk, __fmul_rn(scale, z[j]), A);
                    if (single) {
                        // Step 3a: remember this lane's least E_k; flips wait for all symbols
                        const unsigned long long cand = ((unsigned long long)key_of(E) << 32) | (uint32_t)k;
                        my_best = cand < my_best ? cand : my_best;
                    } else {
                        const uint32_t th = ADAPT ? thr[(t - (int)(sv[j] & kUMask)) & kUMask] : th0;
                        const bool flip = below<PREC>(E, th);
                        if constexpr (kState) {
                            if (flip) st[at + j] = (uint16_t)flip_at(sv[j], xsign != 0u, t);
                        }
                        fmv[j] = __ballot_sync(0xFFFFFFFFu, flip);
                    }
                }
                // Step 3b flips of the group (the single-bit variant flips after the sweep)
                if (lane == 0 && !single) {
                    const uint4 nw = make_uint4(xwv[0] ^ fmv[0], xwv[1] ^ fmv[1], xwv[2] ^ fmv[2], xwv[3] ^ fmv[3]);
                    reinterpret_cast<uint4*>(xw)[g] = nw;
                    if constexpr (CL) {
                        for (int r = 0; split && r < S.size; ++r)
                            if (r != S.rank) reinterpret_cast<uint4*>(peer(xw, r))[g] = nw;
                    }
                }
            }
            if (single && act) atomicMin(bcur + lane, my_best);
        }
        if (ADAPT || !single) break;
        // ---- Step 3a: each decided slot flips its least-E_k symbol (the lowest k among equal
        // values) in every copy of the decision words; every CTA of a split job sees the same
        // minima and takes the same branches ----
        if constexpr (!ADAPT) {
            group_sync();
            if (warp == 0) {
                unsigned long long b = bcur[tid];
                if constexpr (CL) {
                    for (int r = 0; split && r < S.size; ++r) {
                        if (r == S.rank) continue;
                        const unsigned long long o = *peer(bcur + tid, r);
                        b = o < b ? o : b;
                    }
                }
                const bool mine = (todo >> tid) & 1u;
                const float least = value_of((uint32_t)(b >> 32));
                // (with tau at infinity every symbol was evaluated: decided, even if the least is a NaN)
                const bool found = mine && (dense || (b != ~0ull && (least <= tau[tid] || tau[tid] == INFINITY)));
                if (found) {
                    const int k = (int)(uint32_t)b;
                    const bool was_neg = (atomicXor(xw + k, 1u << tid) >> tid) & 1u;
                    if (k >= k_lo && k < k_hi) {
                        const int at = gidx(k - k_lo, tid);
                        if constexpr (SMOOTH) st[at] = (uint16_t)flip_at(st[at], was_neg, round - lane_start[tid]);
                        if constexpr (!dense) {
                            const Job& Jf = job_of(tid);
                            yb[at] = (uint8_t)margin_byte<PREC>(hold<PREC>(read_sample(Jf, lane_frame[tid], k), Jf),
                                                                was_neg ? 0u : 0x80000000u, sym_deg[k - sym_base], Jf);
                        }
                    }
                    if (record) {
                        const int at = (int)atomicAdd(n_flips, 1u);
                        if (at < kFlips) flips[at] = (uint32_t)(k - k_lo) | ((uint32_t)tid << 16);
                    }
                    if constexpr (!dense) tau[tid] = least + kGuess * job_of(tid).scale;
                    if (!split) bcur[tid] = ~0ull;
                } else if (!dense && mine) {
                    tau[tid] = sweep < kSweeps ? tau[tid] + kRaise * job_of(tid).scale : INFINITY;
                }
                // when split, the buffer of the next round (the other CTAs finished reading it
                // before the previous round's closing barrier)
                if (split) best[((round + 1) & 1) * kSlots + tid] = ~0ull;
                const uint32_t left = __ballot_sync(0xFFFFFFFFu, mine && !found);
                if (tid == 0) ctl[5] = left;
            }
            group_sync();
            todo = ctl[5];
            if (todo == 0u) break;
        }
        }
        group_sync();

        // ---- D. the syndromes and counts moved by the flips, when these are few ----
        anew = true;
        if constexpr (!WIDE) {
            // (not in cluster kernels, whose hot code it cost 4 % of the five-code workload: 1.446 -> 1.387 M
            // frames/s; a table's shape is chosen by its measured time.  Not without adaptation: thresholds
            // that do not rise leave few outputs to evaluate -- 20000 frames of the plain decoder at 0 dB take
            // 4.2 ms lazy, 5.0 with every E_k formed -- and the call cost 72 frames of it 6 %)
            if constexpr (!CL && ADAPT) {
                if (!single && (round & kFullEvery) == kFullEvery && __popc(live) > kSlots / 2 &&
                    tally[0] > (uint32_t)(groups_l * kFullMarks) && A.trace_u == nullptr) {
                    round = full_rounds<ADAPT, SMOOTH, ST_SMEM, PREC, CHAIN>(
                        A, ch.jl, ch.slot_e, L.off_icdf, L.off_cnt, L.off_xw, L.off_sw, L.off_thr, L.off_st, chk_cols, sym_chks,
                        sym_deg, sym_groups, ys, st, th0, round);
                    continue;
                }
            }
            const int nf = record ? (int)*n_flips : 0;
            if (record && nf <= few) {
                anew = false;
                // a thread per (flip, check) toggles the check; the old value says which way the counts of
                // its symbols move (kept in the queues' memory)
                uint32_t* moves = reinterpret_cast<uint32_t*>(smem + L.off_queue);
                const int tasks = nf * dv_max;
                for (int i = tid; i < tasks; i += blockDim.x) {
                    const int q = (i * dv_inv) >> 16;           // i / dv_max
                    const uint32_t what = flips[q];
                    const int kl = (int)(what & 0xFFFFu), f = (int)(what >> 16), bit = 2 * (f & 15);
                    const int c = sym_chks[4 * ((size_t)(i - q * dv_max) * sym_groups + sym_g0 + (kl >> 2)) + (kl & 3)];
                    uint32_t move = ~0u;
                    if (c < m) {
                        const uint32_t was = (atomicXor(sw + 2 * c + (f >> 4), 1u << bit) >> bit) & 1u;
                        atomicAdd(unsat_n + f, was ? -1 : 1);
                        move = (uint32_t)c | ((uint32_t)f << 16) | (was << 21);
                    }
                    moves[i] = move;
                }
                __syncthreads();
                // `1 << sg_log` lanes per toggled check, one of its symbols each
                uint32_t* cw = reinterpret_cast<uint32_t*>(cnt);
                const int per = 5 - sg_log;
#pragma unroll 2
                for (int i = (warp << per) + (lane >> sg_log); i < tasks; i += nwarps << per) {
                    const uint32_t move = moves[i];
                    if (move == ~0u) continue;
                    const int c = (int)(move & 0xFFFFu), f = (int)((move >> 16) & 31u), word = cnt_word(f);
                    for (int e = lane & ((1 << sg_log) - 1); e < dc_max; e += 1 << sg_log) {
                        const int k = chk_cols[chk_index(e, c, m)];
                        if (k < n) {
                            const uint32_t one = 1u << (8 * (k & 3) + cnt_shift(f));
                            atomicAdd(cw + (k >> 2) * 16 + word, (move >> 21) & 1u ? 0u - one : one);
                        }
                    }
                }
                __syncthreads();
            }
        }
        ++round;
    }
}

}  // namespace ngdbf
