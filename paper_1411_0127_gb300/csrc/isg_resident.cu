// isg_resident.cu -- sweeps of lattices with few RNG streams, all passes of a
// call in one resident launch.
//
// A lattice with fewer than 16 streams per SM leaves the GPU idle when a warp
// makes a stream's draws (isg_flip_fast.cu): a warp's step of 224 MT19937 draws
// takes about 720 cycles, most of them latency, and every colour pass ends with
// a launch boundary.  Here a block of eight warps shares a stream's draws, and
// the grid stays on the GPU for all passes of the call:
//   * block b owns rpb consecutive rows for the whole launch (MT19937: whole
//     streams), i.e. one or more pieces of streams, whose generator states stay
//     in shared memory between passes;
//   * pass p: the block makes the draws of its rows and leaves their levels in
//     shared memory (two bit streams, or level bytes: take_levels); this needs
//     no other block.  Then it waits (bounded) until the blocks that
//     hold the rows r +- 1, r +- L of its rows have completed pass p - 1,
//     updates its words, one per thread, and publishes its own count.  The
//     blocks that wait for one another have nearly all finished by the time the
//     draws are made, and blocks on one SM overlap each other's waits;
//   * the launch is cooperative: every block is resident, so every count that
//     is waited for comes.
// Draws of a piece, the same values and order as everywhere else:
//   * MT19937: x_{k+624} needs x_k, x_{k+1}, x_{k+397}, so 227 draws can be made
//     at once.  Seven warps make 224 in a step, one draw per thread, with one
//     barrier of the seven warps per step; the stream's words sit in a ring of
//     896 = 4 x 224 words, so that the four phases of a step's addresses are
//     constants and nothing is ever moved.  The tempering and the comparisons
//     of a step run beside the next step's loads.  Draws made past the end of a
//     pass (at most 223) are kept for the next one.  With more than three streams
//     per SM a pair of warps makes a stream's steps instead, four consecutive
//     draws a lane (fewer, wider shared-memory accesses and fewer barriers).
//     MT19937 has no cheap jump, so its streams are not cut into pieces;
//   * MINSTD: draw j of a stream is x 16807^(j+1) mod (2^31 - 1): every thread
//     starts anywhere by one multiplication, four interleaved chains a thread;
//   * Parisi-Rapuano: word n + J of the recurrence x^55 = x^31 + 1 (mod 2^32) is
//     a combination of 55 consecutive words with the coefficients of x^J mod
//     (x^55 - x^31 - 1).  Every warp owns an eighth of the piece and its 64-word
//     window; a jump by a whole pass takes 110 multiply-adds per lane, the price
//     of about ten 32-draw steps.  Of a fresh stream's 61 seed words the last six do
//     not satisfy the recurrence, so a jump by J starts from the last 55 words
//     and uses x^(J-6).
//
// What bounds it: with one MT19937 stream on an SM the chain of a step (loads,
// twist, store, barrier: about 120 cycles for 224 draws, 73 steps a pass) and
// then about 1.8 us of update, publication and wait a pass; with four and more
// streams the two integer pipes, each about 60 % busy (L = 384).  us per colour
// pass, one launch per pass -> resident, calls of 32 sweeps, T = 0.9:
//   L                 64           128          150          256          384
//   MT19937     31.0 -> 6.2  25.0 -> 6.0  37.2 -> 7.0  26.2 -> 13.7  51.2 -> 36.1
//   MINSTD      3.03 -> 2.6  3.23 -> 3.3  5.16 -> 4.1  9.83 -> 7.6   24.9 -> 21.3
//   Par.-Rap.   33.9 -> 3.3  31.8 -> 4.5  43.4 -> 5.2  33.1 -> 12.9  (not used)
#include <algorithm>
#include <cstring>
#include <new>
#include <vector>

#include "isg_bundles.cuh"
#include "isg_levels.cuh"
#include "isg_stream.cuh"

namespace isg {

constexpr int kResThreads = 256, kResWarps = 8;
constexpr int kMtGenWarps = 7, kMtStep = 32 * kMtGenWarps;  // draws of one MT19937 step
constexpr int kMtRing = 4 * kMtStep;                        // 896 >= 624 + 224
constexpr int kLeft = 8;                                    // condition words kept for the next pass (at most 7)
constexpr unsigned kResWaitPolls = 1u << 21;                // about a second with the sleeps
constexpr int kPrSkip = 6, kPrTerms = 55, kPrDigits = 4;

// Coefficients of the Parisi-Rapuano jumps (each x^(J-6) mod x^55 - x^31 - 1):
// 32 (q + 1) 8^i draws, and those of a lattice, a whole pass of a stream and of
// the last stream.
struct PrTo {
    uint32_t to[kPrDigits][7][kPrTerms];
};
struct PrPass {
    uint32_t pass[kPrTerms], last[kPrTerms];
};
struct PrJumps {
    PrTo to;
    PrPass pass;
};
struct NoJumps {};

struct ResidentArgs {
    FlipArgs a;
    int npass;
    int parts, rpb, ncta;          // parts per stream (0: blocks cross streams), rows per block, blocks
    int cw;                        // words of one condition stream
    uint32_t mW, mL, mR;           // n / W, n / L, n / R as umulhi(n, m) (fast_div)
    unsigned long long* done;      // per block: passes completed, the same of all blocks between launches
    unsigned long long* err;       // error word
    unsigned long long stall;      // testing: pass 1 waits for this many passes too many
    unsigned long long* usum;      // not NULL: receives the first pass's unsatisfied bonds before its flips
    const PrPass* jumps;           // Parisi-Rapuano, launches of several lattices
    const uint32_t* rng_in;        // the generator states at the start (levels_kernel: may be a copy of a.rng)
    uint32_t* rng_out;             // minstd_pass_kernel: those at the end, another array
    uint32_t* lv;                  // levels_kernel: where pass 0's levels go (2 cw words a block)
    int64_t lv_pass;               // words between two passes' levels
};

// n / d for n d < 2^32 and m = ceil(2^32 / d) (m d - 2^32 < d, so n m / 2^32 exceeds
// n / d by less than 1 / d); d = 1 has no such 32-bit m.
__device__ __forceinline__ int fast_div(int n, int d, uint32_t m) { return d == 1 ? n : (int)__umulhi((uint32_t)n, m); }

// 16807^e mod (2^31 - 1)
__device__ __forceinline__ uint32_t minstd_power(uint32_t e) {
    uint32_t r = 1, b = kMinstdA;
    for (; e; e >>= 1) {
        if (e & 1u) r = minstd_mulmod(r, b);
        b = minstd_mulmod(b, b);
    }
    return r;
}

// Whether counts [b0, b0 + cnt) (mod ncta) have all reached target; one warp.
__device__ __noinline__ bool res_wait(const unsigned long long* done, unsigned long long* err, int b0, int cnt,
                                      int ncta, unsigned long long target, int lane) {
    bool ok = true;
    for (int j0 = 0; j0 < cnt && ok; j0 += 32) {
        bool mine = true;
        if (j0 + lane < cnt) {
            int b = b0 + j0 + lane;
            b = b >= ncta ? b - ncta : b;
            mine = false;
            for (unsigned it = 0; it < kResWaitPolls; ++it) {
                if (ld_acquire_u64(done + b) >= target) {
                    mine = true;
                    break;
                }
                if ((it & 63u) == 63u) {
                    if (*(volatile const unsigned long long*)err != 0ull) break;
                    __nanosleep(it < 4096u ? 32 : 512);
                }
            }
        }
        ok = __all_sync(kFull, mine);
    }
    if (!ok && lane == 0) atomicExch(err, 1ull);
    return ok;
}

// Levels of one 32-draw block: one word of each condition stream, stored by
// lanes 0 (lo) and 1 (hi); `at` is the lane's shared-window address of its word.
__device__ __forceinline__ void block_cond(uint32_t d, const Cmp& cm, uint32_t at, int lane) {
    const uint32_t lo = __ballot_sync(kFull, level_lo(d, cm));
    const uint32_t hi = __ballot_sync(kFull, d < cm.c2);
    const uint32_t v = lane == 0 ? lo : hi;
    asm volatile("{\n\t.reg .pred p;\n\tsetp.lt.s32 p, %2, 2;\n\t@p st.shared.u32 [%0], %1;\n\t}"
                 :
                 : "r"(at), "r"(v), "r"(lane)
                 : "memory");
}

// The same of four consecutive blocks: four words at shared-window address `at`
// and four at at + hi.  No draw below thr2 in most of them: one comparison a draw.
__device__ __forceinline__ void quad_cond(const uint32_t (&d)[4], const Cmp& cm, uint32_t at, int hi, int lane) {
    uint32_t l[4], h[4];
    const uint32_t dmin = min(min3(d[0], d[1], d[2]), d[3]);
    if (__any_sync(kFull, dmin < cm.c2)) {
        level_ballots<4>(d, cm, l, h);
    } else {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            l[q] = __ballot_sync(kFull, d[q] < cm.c1);
            h[q] = 0u;
        }
    }
    st_shared_lane0(at, l[0], l[1], l[2], l[3], lane);
    st_shared_lane0(at + hi, h[0], h[1], h[2], h[3], lane);
}

// ------------------------------------------------------------- MT19937 ---
// One step in phase PH (k mod 896 = 224 PH): thread tid of seven warps makes
// x_{k+624+tid}.  A step reads words that exist before it and writes slots of
// words older than x_k, so the barrier between steps is the only one it needs.
// i1, im, iw are the wrapped indices of the phases where a thread-dependent wrap
// occurs.  While the step's loads are on their way, the previous step's draw is
// tempered and that of the step before it compared (two chains that do not
// depend on each other).
struct TeamStep {
    uint32_t* ring;
    int tid, lane, i1, im, iw;
    uint32_t at;  // address of the next condition word (block_cond)
};

// EMIT: 0 the first step, 1 the second (`raw` to temper, nothing to compare), 2 any later one
template <int PH, int EMIT>
__device__ __forceinline__ void mt_team_step(TeamStep& q, uint32_t& raw, uint32_t& d, const Cmp& cm, const MtMul& k) {
    const uint32_t a = q.ring[kMtStep * PH + q.tid];
    const uint32_t b = q.ring[PH == 3 ? q.i1 : kMtStep * PH + q.tid + 1];
    const uint32_t m = q.ring[PH == 2 ? q.im : (kMtStep * PH + kMtM) % kMtRing + q.tid];
    if (EMIT == 2) {
        block_cond(d, cm, q.at, q.lane);
        q.at += 4 * kMtGenWarps;
    }
    if (EMIT >= 1) d = mt_temper_mul(raw, k);
    raw = mt_twist(a, b, m, k);
    q.ring[PH == 1 ? q.iw : (kMtStep * PH + kMtN) % kMtRing + q.tid] = raw;
    asm volatile("bar.sync 1, %0;" ::"n"(kMtStep) : "memory");
}

// f(phase as a compile-time constant)
template <class F>
__device__ __forceinline__ void with_phase(int ph, F&& f) {
    if (ph == 0) f(std::integral_constant<int, 0>{});
    else if (ph == 1) f(std::integral_constant<int, 1>{});
    else if (ph == 2) f(std::integral_constant<int, 2>{});
    else f(std::integral_constant<int, 3>{});
}

// n steps starting in phase `ph`; block j of step i goes to condition word
// first + 7 i + j.  Warps 0..6.
__device__ __forceinline__ void mt_team_run(uint32_t* ring, int ph, int n, uint32_t* cond, int cw, int first,
                                            const Cmp& cm, const MtMul& k) {
    if (n <= 0) return;
    TeamStep q;
    q.ring = ring;
    q.tid = threadIdx.x;
    q.lane = q.tid & 31;
    q.i1 = q.tid == kMtStep - 1 ? 0 : 3 * kMtStep + q.tid + 1;
    q.im = 2 * kMtStep + kMtM + q.tid;
    q.im = q.im >= kMtRing ? q.im - kMtRing : q.im;
    q.iw = kMtStep + kMtN + q.tid;
    q.iw = q.iw >= kMtRing ? q.iw - kMtRing : q.iw;
    q.at = (uint32_t)__cvta_generic_to_shared(cond + first + (q.tid >> 5) + (q.lane == 0 ? 0 : cw));
    uint32_t raw = 0, d = 0;
    with_phase(ph, [&](auto P) { mt_team_step<decltype(P)::value, 0>(q, raw, d, cm, k); });
    if (n > 1) {
        ph = (ph + 1) & 3;
        with_phase(ph, [&](auto P) { mt_team_step<decltype(P)::value, 1>(q, raw, d, cm, k); });
        ph = (ph + 1) & 3;
        n -= 2;
        for (; n > 0 && ph != 0; --n, ph = (ph + 1) & 3)
            with_phase(ph, [&](auto P) { mt_team_step<decltype(P)::value, 2>(q, raw, d, cm, k); });
        for (; n >= 4; n -= 4) {
            mt_team_step<0, 2>(q, raw, d, cm, k);
            mt_team_step<1, 2>(q, raw, d, cm, k);
            mt_team_step<2, 2>(q, raw, d, cm, k);
            mt_team_step<3, 2>(q, raw, d, cm, k);
        }
        for (; n > 0; --n, ph = (ph + 1) & 3)
            with_phase(ph, [&](auto P) { mt_team_step<decltype(P)::value, 2>(q, raw, d, cm, k); });
        block_cond(d, cm, q.at, q.lane);
        q.at += 4 * kMtGenWarps;
    }
    block_cond(mt_temper_mul(raw, k), cm, q.at, q.lane);
}

// Two warps make the 224 draws of a step, four consecutive ones a lane (28 lanes
// of each), as level bytes: byte `first` + 56 i + quad for step i.  Lane 28 loads
// the quad after the warp's last, so that the word after a lane's quad comes from
// the next lane.  `bar` is the pair's named barrier; of a block that is one pair
// (ONE) it is barrier 1, a constant: a kernel with a barrier number in a register
// is given all 16, and an SM has 64, so no more than four such blocks.
struct PairStep {
    uint32_t* ring;
    int q4, bar;         // first word of the lane's quad, barrier
    int a, m, w;         // wrapped indices (a of phase 3, m of phase 2, w of phase 1)
    bool mine;           // the lane's quad is its own to store
    unsigned char* at;   // the lane's next level byte
};

template <int PH, bool EMIT, bool ONE>
__device__ __forceinline__ void mt_pair_step(PairStep& q, uint32_t (&raw)[4], const Cmp& cm, const Cmp4& c4,
                                             const MtMul& k) {
    constexpr int b0 = kMtStep * PH, bm = (kMtStep * PH + kMtM - 1) % kMtRing, bw = (kMtStep * PH + kMtN) % kMtRing;
    const uint4 a = *(const uint4*)(q.ring + (PH == 3 ? q.a : b0 + q.q4));
    const uint4 m = *(const uint4*)(q.ring + (PH == 2 ? q.m : bm + q.q4));
    LevelHalf h;
    if (EMIT) h = mt_level_begin(raw, c4, k);
    const uint32_t an = __shfl_down_sync(kFull, a.x, 1), mn = __shfl_down_sync(kFull, m.x, 1);
    mt_twist4(a, an, m, mn, raw, k);
    if (q.mine) *(uint4*)(q.ring + (PH == 1 ? q.w : bw + q.q4)) = make_uint4(raw[0], raw[1], raw[2], raw[3]);
    if (EMIT) {
        const uint32_t byte = mt_level_finish(h, cm, c4);
        if (q.mine) *q.at = (unsigned char)byte;
        q.at += kMtStep / 4;
    }
    if (ONE) asm volatile("bar.sync 1, 64;" ::: "memory");
    else asm volatile("bar.sync %0, 64;" ::"r"(q.bar) : "memory");
}

template <bool ONE>
__device__ __forceinline__ void mt_pair_run(uint32_t* ring, int ph, int n, unsigned char* bytes, int half_of_pair,
                                            int bar, const Cmp& cm, const MtMul& k) {
    if (n <= 0) return;
    const int quad = 28 * half_of_pair + min((int)(threadIdx.x & 31), 28);
    const Cmp4 c4 = cmp4_of(cm);
    PairStep q;
    q.ring = ring;
    q.q4 = 4 * quad;
    q.bar = bar;
    auto wrap = [](int i) { return i >= kMtRing ? i - kMtRing : i; };
    q.a = wrap(3 * kMtStep + q.q4);
    q.m = wrap(2 * kMtStep + kMtM - 1 + q.q4);
    q.w = wrap(kMtStep + kMtN + q.q4);
    q.mine = (threadIdx.x & 31) < 28;
    q.at = bytes + quad;
    uint32_t raw[4] = {};
    with_phase(ph, [&](auto P) { mt_pair_step<decltype(P)::value, false, ONE>(q, raw, cm, c4, k); });
    ph = (ph + 1) & 3;
    --n;
    for (; n > 0 && ph != 0; --n, ph = (ph + 1) & 3)
        with_phase(ph, [&](auto P) { mt_pair_step<decltype(P)::value, true, ONE>(q, raw, cm, c4, k); });
    for (; n >= 4; n -= 4) {
        mt_pair_step<0, true, ONE>(q, raw, cm, c4, k);
        mt_pair_step<1, true, ONE>(q, raw, cm, c4, k);
        mt_pair_step<2, true, ONE>(q, raw, cm, c4, k);
        mt_pair_step<3, true, ONE>(q, raw, cm, c4, k);
    }
    for (; n > 0; --n, ph = (ph + 1) & 3)
        with_phase(ph, [&](auto P) { mt_pair_step<decltype(P)::value, true, ONE>(q, raw, cm, c4, k); });
    const uint32_t byte = mt_level_finish(mt_level_begin(raw, c4, k), cm, c4);
    if (q.mine) *q.at = (unsigned char)byte;
}

// ------------------------------------------------------ Parisi-Rapuano ---
// Words ira[n+J-64+m], m = lane and lane + 32, from X[i] = ira[n-64+i] (i < 128)
// and the coefficients c of x^(J-6): ira[n+J-64+m] = sum c_i ira[n-58+m+i].
__device__ __forceinline__ void pr_jump(const uint32_t* X, const uint32_t* c, int lane, uint32_t& ya, uint32_t& yb) {
    uint32_t s0 = 0, s1 = 0;
#pragma unroll 11
    for (int i = 0; i < kPrTerms; ++i) {
        const uint32_t ci = c[i];
        s0 += ci * X[lane + kPrSkip + i];
        s1 += ci * X[lane + 32 + kPrSkip + i];
    }
    ya = s0;
    yb = s1;
}

// 32-draw blocks of one warp's share of a piece of D draws, a multiple of 4
__device__ __forceinline__ int pr_share(int D) { return (D + 128 * kResWarps - 1) / (128 * kResWarps) * 4; }

// The window (a, b) and the two steps after it as 128 words in X; (a, b) ends
// two steps on.
__device__ __forceinline__ void pr_span(uint32_t* X, uint32_t& a, uint32_t& b, int lane, uint32_t& d0, uint32_t& d1) {
    X[lane] = a;
    X[32 + lane] = b;
    d0 = pr_warp_step(a, b, lane, 32);
    X[64 + lane] = b;
    d1 = pr_warp_step(a, b, lane, 32);
    X[96 + lane] = b;
    __syncwarp();
}

// ---------------------------------------------------------------- kernel ---
// Shared memory of a block (words): the levels of a pass, 2 cw per stream whose
// draws are made at once; Parisi-Rapuano: 8 spans of 128; then per stream
// MT19937: ring 896 (rings first, then the kept words 2 kLeft of each); MINSTD:
// 4; Parisi-Rapuano: 8 windows of 64.
template <int KIND>
__host__ __device__ constexpr int res_stream_words() {
    return KIND == ISG_RNG_MT19937 ? kMtRing + 2 * kLeft : (KIND == ISG_RNG_PARISI_RAPUANO ? kResWarps * 64 : 4);
}
template <int KIND>
__host__ __device__ constexpr int res_fixed_words() {
    return KIND == ISG_RNG_PARISI_RAPUANO ? kResWarps * 128 : 0;
}

// PAIRS: streams of a block whose draws are made by a pair of warps each (MT19937;
// the block has 64 PAIRS threads, levels are bytes); 0: blocks of 256 threads
// that take their streams one by one (MT19937: seven warps; levels are lo / hi
// bit streams).  MINB: resident blocks per SM that the registers allow.
// With LEVELS (one piece a block) the levels of each pass are only written out,
// for other kernels to use, and nothing is updated or waited for.
// With APART (MINSTD) the launch is one pass, of colour a.c, that waits for the
// launch before it; its blocks wait for none of its own, since the states at the
// end go to another array than those that other blocks may still have to read.
// ONE: see PairStep.
template <typename Word, int KIND, int PAIRS, bool LEVELS = false, bool APART = false, bool ONE = PAIRS == 1>
__device__ __forceinline__ void resident_block(const ResidentArgs& A, const StreamConst& K, const PrTo* J,
                                               const PrPass* JP, int bid) {
    extern __shared__ __align__(16) uint32_t smem[];
    __shared__ int s_ok;
    constexpr int w = 8 * sizeof(Word);
    constexpr bool kMT = KIND == ISG_RNG_MT19937;
    constexpr int NS = PAIRS ? PAIRS : 1, kThreads = PAIRS ? 64 * PAIRS : kResThreads;
    constexpr int kSW = kMT ? kMtRing : res_stream_words<KIND>();
    const FlipArgs& a = A.a;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int L = a.L, half = a.half, W = a.W, rows = (int)a.rows, R = (int)a.R, S = (int)a.S, cw = A.cw;
    uint32_t* cond = smem;
    uint32_t* fixed = smem + 2 * cw * NS;
    uint32_t* state = fixed + res_fixed_words<KIND>();
    uint32_t* kept = state + NS * kMtRing;  // MT19937
    const Cmp cm = cmp_of(a);

    // this block's rows [rb, re): pieces of the streams t0 .. t0 + nst - 1
    auto block_of = [&](int r) { return A.parts ? r / R * A.parts + r % R / A.rpb : r / A.rpb; };
    const int rb = A.parts ? min(rows, bid / A.parts * R + bid % A.parts * A.rpb) : bid * A.rpb;
    const int re = min(rows, A.parts ? min(rb + A.rpb, (bid / A.parts + 1) * R) : rb + A.rpb);
    if (rb >= re) {  // an empty part of a short last stream
        if (!LEVELS && !APART && tid == 0)
            st_release_u64(A.done + bid, A.done[bid] + (unsigned long long)A.npass);
        return;
    }
    // Passes completed by the earlier launches, in the warps that wait and publish.
    // Read here, not passed: a launch captured into a graph and replayed then
    // starts from the counts it finds.  (From a register: from shared memory L = 64
    // MT19937 took 6.3 instead of 6.2 us a pass.)
    unsigned long long base = 0;
    if (!LEVELS && !APART && (wid == 0 || wid == kThreads / 32 - 1)) base = A.done[bid];
    const int t0 = rb / R, nst = (re - 1) / R - t0 + 1;
    auto stream_rows = [&](int t) { return min(rows, (t + 1) * R) - t * R; };
    // the blocks holding rows rb - L .. re - 1 + L (cyclic)
    int dep0 = 0, depn = A.ncta;
    if (re - rb + 2 * L < rows) {
        const int lo = rb - L, hi = re - 1 + L;
        dep0 = block_of(lo < 0 ? lo + rows : lo);
        depn = (block_of(hi >= rows ? hi - rows : hi) - dep0 + A.ncta) % A.ncta + 1;
    }

    // generator states into shared memory
    uint32_t pw = 0, step1024 = 0;  // MINSTD: 16807^(first draw of this thread + 1), 16807^1024
    if (APART) {
        // what does not come from the launch before this one is made while that one ends
        for (int i = tid; i < 2 * nst; i += kThreads) {
            const int t = t0 + (i >> 1);
            state[(i >> 1) * kSW + 2 + (i & 1)] =
                minstd_power((uint32_t)((i & 1 ? stream_rows(t) : max(rb, t * R) - t * R) * half));
        }
        pw = minstd_power((uint32_t)(wid * 128 + lane + 1));
        step1024 = minstd_power(1024u);
        __syncthreads();
        asm volatile("griddepcontrol.wait;" ::: "memory");
        asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
        for (int s = tid; s < nst; s += kThreads) {
            const uint32_t x = A.rng_in[t0 + s];
            state[s * kSW] = minstd_mulmod(x, state[s * kSW + 2]);
            if ((t0 + s) * R >= rb) A.rng_out[t0 + s] = minstd_mulmod(x, state[s * kSW + 3]);
        }
    }
    for (int s = 0; !APART && s < nst; ++s) {
        const int64_t t = t0 + s;
        uint32_t* st = state + s * kSW;
        if (kMT) {
            const int p = (int)a.rng_pos[t];
            for (int j = tid; j < kMtN; j += kThreads) st[j] = A.rng_in[t * kMtN + (p + j >= kMtN ? p + j - kMtN : p + j)];
        } else if (KIND == ISG_RNG_MINSTD) {
            if (tid == 0) {
                st[0] = minstd_mulmod(A.rng_in[t], minstd_power((uint32_t)((max(rb, (int)t * R) - (int)t * R) * half)));
                st[1] = minstd_power((uint32_t)(stream_rows((int)t) * half));  // a whole pass
            }
        } else {
            if constexpr (KIND == ISG_RNG_PARISI_RAPUANO) {
                const int r0 = max(rb, (int)t * R), D = (min(re, (int)(t + 1) * R) - r0) * half;
                const int n = (r0 - (int)t * R) * half + 32 * wid * pr_share(D);  // draws before this warp's first
                uint32_t xa, xb, d0, d1;
                pr_load(A.rng_in + t * kPrN, xa, xb, lane);
                uint32_t* X = fixed + wid * 128;
                if (n & 31) pr_warp_step(xa, xb, lane, n & 31);
                for (int i = 0, q = n >> 5; q; ++i, q >>= 3) {
                    if (!(q & 7)) continue;
                    pr_span(X, xa, xb, lane, d0, d1);
                    pr_jump(X, J->to[i][(q & 7) - 1], lane, xa, xb);
                    __syncwarp();
                }
                st[wid * 64 + lane] = xa;
                st[wid * 64 + 32 + lane] = xb;
            }
        }
    }
    if (KIND == ISG_RNG_MINSTD && !APART) {
        pw = minstd_power((uint32_t)(wid * 128 + lane + 1));
        step1024 = minstd_power(1024u);
    }
    __syncthreads();

    int dEsum = 0, usum = 0;
    bool ok = true;
    const int ngroups = PAIRS ? 1 : nst;
    for (int p = 0; p < A.npass && ok; ++p) {
        const int c = APART ? a.c : p & 1;
        for (int s = 0; s < ngroups; ++s) {
            const int t = t0 + s;
            // the rows of this group (all of the block's, or a piece's) and their draws
            const int grb = PAIRS ? rb : max(rb, t * R), gre = PAIRS ? re : min(re, (t + 1) * R);
            const int D = (gre - grb) * half;
            uint32_t* st = state + s * kSW;
            int off0 = 0;           // bit of the condition streams that is the group's first draw
            int left = 0, keep = 0; // MT19937: words of levels made, first one the next pass needs
            if constexpr (kMT && !PAIRS) {
                const int P0 = p * D, n0 = (P0 + kMtStep - 1) / kMtStep, n1 = (P0 + D + kMtStep - 1) / kMtStep;
                off0 = P0 & 31;
                left = kMtGenWarps * n0 - (P0 >> 5);
                keep = (P0 + D) / 32 - (P0 >> 5);
                if (wid == 0 && (lane & (kLeft - 1)) < left && lane < 2 * kLeft)
                    cond[(lane < kLeft ? 0 : cw) + (lane & (kLeft - 1))] = kept[lane];
                if (wid < kMtGenWarps) mt_team_run(st, n0 & 3, n1 - n0, cond, cw, left, cm, K.mul);
                left = kMtGenWarps * n1 - (P0 >> 5);
            } else if constexpr (kMT) {
                // warps 2 s2 and 2 s2 + 1 make stream s2's draws: a scheduler's warps belong to different streams
                const int s2 = wid >> 1;
                if (s2 < nst) {
                    const int P0 = p * stream_rows(t0 + s2) * half, P1 = P0 + stream_rows(t0 + s2) * half;
                    const int n0 = (P0 + kMtStep - 1) / kMtStep, n1 = (P1 + kMtStep - 1) / kMtStep;
                    uint32_t* lv = cond + s2 * 2 * cw;
                    left = kMtStep / 16 * n0 - (P0 >> 4);
                    keep = (P1 >> 4) - (P0 >> 4);
                    if ((wid & 1) == 0 && lane < left) lv[lane] = kept[s2 * 2 * kLeft + lane];
                    mt_pair_run<ONE>(state + s2 * kSW, n0 & 3, n1 - n0, (unsigned char*)(lv + left), wid & 1,
                                     1 + s2, cm, K.mul);
                    left = kMtStep / 16 * n1 - (P0 >> 4);
                }
            } else if constexpr (KIND == ISG_RNG_MINSTD) {
                uint32_t x[4];
                x[0] = minstd_mulmod(st[0], pw);
#pragma unroll
                for (int q = 1; q < 4; ++q) x[q] = minstd_mulmod(x[q - 1], K.a32);
                const int nq = (D + 127) >> 7;
                const uint32_t cs = (uint32_t)__cvta_generic_to_shared(cond);
                for (int j = wid; j < nq; j += kResWarps) {
                    quad_cond(x, cm, cs + 16 * j, 4 * cw, lane);
#pragma unroll
                    for (int q = 0; q < 4; ++q) x[q] = minstd_mulmod(x[q], step1024);
                }
            } else {
                const int b0 = wid * pr_share(D), nb = min(pr_share(D), ((D + 31) >> 5) - b0);
                if (nb > 0) {
                    uint32_t xa = st[wid * 64 + lane], xb = st[wid * 64 + 32 + lane], d0, d1, ya, yb;
                    uint32_t* X = fixed + wid * 128;
                    pr_span(X, xa, xb, lane, d0, d1);
                    pr_jump(X, t == S - 1 ? JP->last : JP->pass, lane, ya, yb);
                    st[wid * 64 + lane] = ya;
                    st[wid * 64 + 32 + lane] = yb;
                    const uint32_t cs = (uint32_t)__cvta_generic_to_shared(cond + b0);
                    for (int j = 0; j < nb; j += 4) {
                        uint32_t d[4] = {d0, d1, 0, 0};
#pragma unroll
                        for (int q = 0; q < 4; ++q)
                            if (q >= 2 || j > 0) d[q] = pr_warp_step(xa, xb, lane, 32);
                        quad_cond(d, cm, cs + 4 * j, 4 * cw, lane);
                    }
                }
            }
            if constexpr (LEVELS) {
                __syncthreads();
                // the words that hold the pass's draws, and what a window of a last word reads behind them
                uint32_t* to = A.lv + p * A.lv_pass + (int64_t)bid * 2 * cw;
                if constexpr (PAIRS) {
                    for (int i = tid; i < (D + 31) / 16 + 1; i += kThreads) to[i] = cond[i];
                } else {
                    for (int i = tid; i < 2 * ((D + 63) / 32 + 1); i += kThreads)
                        to[(i & 1) * cw + (i >> 1)] = cond[(i & 1) * cw + (i >> 1)];
                }
            }
            if (!LEVELS && wid == kThreads / 32 - 1 && s == 0) {
                bool go = *(volatile const unsigned long long*)A.err == 0ull;
                if (!APART && go && p > 0)
                    go = res_wait(A.done, A.err, dep0, depn, A.ncta,
                                  base + (unsigned long long)p + (p == 1 ? A.stall : 0ull), lane);
                if (lane == 0) s_ok = go;
            }
            if (!LEVELS) {
                __syncthreads();
                ok = s_ok != 0;
                if (!ok) break;
            }
            const int nw = LEVELS ? 0 : (gre - grb) * W;
            for (int i = tid; i < nw; i += kThreads) {
                const int j = fast_div(i, W, A.mW), k = i - j * W, r = grb + j;
                const int z = fast_div(r, L, A.mL), y = r - z * L;
                WordIn<Word> q;
                word_load<Word, true>(a, c, r, y, z, k, q);
                Word lo, hi;
                if constexpr (PAIRS) {
                    const int s2 = fast_div(j, R, A.mR), P0 = p * stream_rows(t0 + s2) * half;
                    take_levels<Word>(cond + s2 * 2 * cw, (P0 & 15) + (j - s2 * R) * half + k * w, lo, hi);
                } else {
                    lo = take_bits<Word>(cond, off0 + j * half + k * w);
                    hi = take_bits<Word>(cond + cw, off0 + j * half + k * w);
                }
                if (p == 0 && A.usum) word_flip<Word>(a, c, q, k, lo, hi, dEsum, &usum);
                else word_flip<Word>(a, c, q, k, lo, hi, dEsum);
            }
            // MT19937: keep the levels of draws past the end of the pass
            if constexpr (kMT && !PAIRS) {
                if (wid == 0 && lane < 2 * kLeft && keep + (lane & (kLeft - 1)) < left)
                    kept[lane] = cond[(lane < kLeft ? 0 : cw) + keep + (lane & (kLeft - 1))];
            } else if constexpr (kMT) {
                if ((wid & 1) == 0 && (wid >> 1) < nst && keep + lane < left)
                    kept[wid * kLeft + lane] = cond[wid * cw + keep + lane];
            }
            if (KIND == ISG_RNG_MINSTD && !APART && tid == 0) st[0] = minstd_mulmod(st[0], st[1]);
            __syncthreads();
        }
        if (!LEVELS && !APART && ok && tid == kThreads - 32) {  // every thread's stores came before the barrier
            __threadfence();
            st_release_u64(A.done + bid, base + (unsigned long long)p + 1ull);
        }
    }

    if (!APART) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    // a block that gave up leaves the count of one that did not (the error word is set)
    if (!LEVELS && !APART && !ok && tid == 0) st_release_u64(A.done + bid, base + (unsigned long long)A.npass);
    // generator states back, by the block that holds a stream's first rows, once
    // the blocks with its other rows have read theirs
    if (ok && !APART) {
        const int tl = t0 + nst - 1, rl = min(rows, (tl + 1) * R);
        if (!LEVELS && tl * R >= rb && rl > re) {
            if (wid == 0) {
                const bool go = res_wait(A.done, A.err, bid + 1, block_of(rl - 1) - bid, A.ncta, base + 1ull, lane);
                if (lane == 0) s_ok = go;
            }
            __syncthreads();
            ok = s_ok != 0;
        }
        for (int s = 0; s < nst && ok; ++s) {
            if ((t0 + s) * R < rb) continue;
            const int64_t t = t0 + s;
            uint32_t* st = state + s * kSW;
            if (kMT) {
                const int K = A.npass * (stream_rows((int)t) * half);
                const int pos = ((int)a.rng_pos[t] + K) % kMtN;
                for (int j = tid; j < kMtN; j += kThreads)
                    a.rng[t * kMtN + (pos + j >= kMtN ? pos + j - kMtN : pos + j)] = st[(K + j) % kMtRing];
                __syncthreads();
                if (tid == 0) a.rng_pos[t] = (uint32_t)pos;
            } else if (KIND == ISG_RNG_MINSTD) {
                if (tid == 0) a.rng[t] = st[0];
            } else if (wid == 0) {
                pr_store(a.rng + t * kPrN, st[lane], st[32 + lane], lane);
            }
        }
    }
    if constexpr (!LEVELS) {
        for (int sh = 16; sh; sh >>= 1) dEsum += __shfl_xor_sync(kFull, dEsum, sh);
        if (lane == 0 && dEsum != 0) atomicAdd((unsigned long long*)a.dE, (unsigned long long)(long long)dEsum);
        if (A.usum) {
            for (int sh = 16; sh; sh >>= 1) usum += __shfl_xor_sync(kFull, usum, sh);
            if (lane == 0 && usum != 0) atomicAdd(A.usum, (unsigned long long)usum);
        }
    }
}

template <typename Word, int KIND, int PAIRS, int MINB, class Jumps>
__global__ void __launch_bounds__(PAIRS ? 64 * PAIRS : kResThreads, MINB)
    resident_kernel(const __grid_constant__ ResidentArgs A, const __grid_constant__ StreamConst K,
                    const __grid_constant__ Jumps J) {
    if constexpr (KIND == ISG_RNG_PARISI_RAPUANO) resident_block<Word, KIND, PAIRS>(A, K, &J.to, &J.pass, blockIdx.x);
    else resident_block<Word, KIND, PAIRS>(A, K, nullptr, nullptr, blockIdx.x);
}

// One MINSTD pass as a launch of its own.
template <typename Word>
__global__ void __launch_bounds__(kResThreads, 4)
    minstd_pass_kernel(const __grid_constant__ ResidentArgs A, const __grid_constant__ StreamConst K) {
    resident_block<Word, ISG_RNG_MINSTD, 0, false, true>(A, K, nullptr, nullptr, blockIdx.x);
}

// Several lattices (64-bit words) in one launch: block b is block blocks[b].y of
// lattice blocks[b].x.  npass > 0 takes the place of the table's.  Passes [first,
// first + kResidentPasses) of them are this launch's; a lattice with no pass there
// has nothing to do (all of its blocks leave, so its counts stay equal).  Up to four
// blocks of one pair an SM name their barrier by a register all the same, and so
// keep an SM's 64 for themselves: a server sweeps its three generator kinds side by
// side, and with blocks of the others beside them, whose waits poll, 24 jobs took up
// to 19 % longer (32.7 against 38.2 ms).
template <int KIND, int PAIRS, int MINB, class To>
__global__ void __launch_bounds__(PAIRS ? 64 * PAIRS : kResThreads, MINB)
    resident_set_kernel(const ResidentArgs* tab, const int2* blocks, int npass, int first,
                        const __grid_constant__ StreamConst K, const __grid_constant__ To J) {
    __shared__ ResidentArgs A;
    static_assert(sizeof(ResidentArgs) % 4 == 0, "copied by words");
    const int2 e = blocks[blockIdx.x];
    for (unsigned i = threadIdx.x; i < sizeof(ResidentArgs) / 4; i += blockDim.x)
        ((uint32_t*)&A)[i] = ((const uint32_t*)(tab + e.x))[i];
    __syncthreads();
    const int n = (npass > 0 ? npass : A.npass) - first;
    if (n <= 0) return;
    __syncthreads();
    if (threadIdx.x == 0) A.npass = min(n, kResidentPasses);
    __syncthreads();
    if constexpr (KIND == ISG_RNG_PARISI_RAPUANO) resident_block<uint64_t, KIND, PAIRS>(A, K, &J, A.jumps, e.y);
    else resident_block<uint64_t, KIND, PAIRS, false, false, PAIRS == 1 && MINB != 4>(A, K, nullptr, nullptr, e.y);
}

// The levels of npass passes of one generator alone (isg_amsc.cu).
template <int KIND, int PAIRS, class Jumps>
__global__ void __launch_bounds__(PAIRS ? 64 * PAIRS : kResThreads, PAIRS ? 14 : 4)
    levels_kernel(const __grid_constant__ ResidentArgs A, const __grid_constant__ StreamConst K,
                  const __grid_constant__ Jumps J) {
    if constexpr (KIND == ISG_RNG_PARISI_RAPUANO)
        resident_block<uint32_t, KIND, PAIRS, true>(A, K, &J.to, &J.pass, blockIdx.x);
    else
        resident_block<uint32_t, KIND, PAIRS, true>(A, K, nullptr, nullptr, blockIdx.x);
}

// ------------------------------------------------------------------ host ---
// r = r q mod (x^55 - x^31 - 1), coefficients mod 2^32
static void pr_mul(uint32_t* r, const uint32_t* q) {
    uint32_t t[2 * kPrTerms - 1] = {};
    for (int i = 0; i < kPrTerms; ++i)
        for (int j = 0; j < kPrTerms; ++j) t[i + j] += r[i] * q[j];
    for (int i = 2 * kPrTerms - 2; i >= kPrTerms; --i) {
        t[i - kPrTerms] += t[i];
        t[i - 24] += t[i];
    }
    memcpy(r, t, kPrTerms * sizeof(uint32_t));
}

// c = c x mod (x^55 - x^31 - 1)
static void pr_shift(uint32_t* c) {
    const uint32_t top = c[kPrTerms - 1];
    memmove(c + 1, c, (kPrTerms - 1) * sizeof(uint32_t));
    c[0] = top;
    c[31] += top;
}

// Coefficients of x^(J - 6), 6 <= J < 2^32.
static void pr_coefficients(uint64_t J, uint32_t* c) {
    memset(c, 0, kPrTerms * sizeof(uint32_t));
    c[0] = 1;
    const uint64_t e = J - kPrSkip;
    bool any = false;
    for (int b = 31; b >= 0; --b) {
        if (any) pr_mul(c, c);
        if ((e >> b) & 1) {
            pr_shift(c);
            any = true;
        }
    }
}

// c = the coefficients of a jump by the sum of a's and b's: x^(I+J-6) = x^(I-6) x^(J-6) x^6
static void pr_combine(const uint32_t* a, const uint32_t* b, uint32_t* c) {
    uint32_t t[kPrTerms];
    memcpy(t, a, sizeof t);
    pr_mul(t, b);
    for (int q = 0; q < kPrSkip; ++q) pr_shift(t);
    memcpy(c, t, sizeof t);
}

// The coefficients that do not depend on the lattice, made once (about 70 us).
static const PrTo& pr_to() {
    static const PrTo table = [] {
        PrTo J;
        for (int i = 0; i < kPrDigits; ++i) {
            if (i == 0) pr_coefficients(32, J.to[0][0]);
            else pr_combine(J.to[i - 1][6], J.to[i - 1][0], J.to[i][0]);
            for (int q = 1; q < 7; ++q) pr_combine(J.to[i][q - 1], J.to[i][0], J.to[i][q]);
        }
        return J;
    }();
    return table;
}

static void pr_pass(const isg_sim* h, PrPass& P) {
    pr_coefficients((uint64_t)(h->R * h->half), P.pass);
    pr_coefficients((uint64_t)((h->rows - (h->S - 1) * h->R) * h->half), P.last);
}

// How a lattice is laid out over the blocks of a resident launch.
struct ResidentLayout {
    int parts = 0, rpb = 0, ncta = 0, cw = 0;
    size_t smem = 0;
};

// MT19937: `pairs` (or one) whole streams a block; else at most `cap` blocks:
// parts of a stream, or, with more streams than blocks or `even`, an even share
// of the rows, at least 64 words each.
static ResidentLayout layout_of(const isg_sim* h, int pairs, int64_t cap, bool even = false) {
    ResidentLayout P;
    const bool mt = h->kind == ISG_RNG_MT19937;
    int64_t rpb = h->R * (pairs ? pairs : 1);
    if (!mt && (even || h->S > cap)) rpb = std::max<int64_t>((64 + h->W - 1) / h->W, (h->rows + cap - 1) / cap);
    if (!mt && !even && h->S <= cap) {
        const int64_t least = (64 + h->W - 1) / h->W;
        const int64_t parts = std::max<int64_t>(1, std::min((h->R + least - 1) / least, cap / h->S));
        rpb = (h->R + parts - 1) / parts;
        P.parts = (int)((h->R + rpb - 1) / rpb);
    }
    P.rpb = (int)std::min<int64_t>(rpb, h->rows);
    P.ncta = P.parts ? (int)(h->S * P.parts) : (int)((h->rows + P.rpb - 1) / P.rpb);
    const int pieces = mt ? (pairs ? pairs : 1) : (int)((P.rpb + h->R - 2) / h->R + 1);
    const int D = (int)std::min<int64_t>(P.rpb, h->R) * h->half;
    P.cw = (D / 32 + 20 + 3) / 4 * 4;
    const int stream = mt ? res_stream_words<ISG_RNG_MT19937>()
                          : (h->kind == ISG_RNG_MINSTD ? res_stream_words<ISG_RNG_MINSTD>()
                                                       : res_stream_words<ISG_RNG_PARISI_RAPUANO>());
    const int fixed = h->kind == ISG_RNG_PARISI_RAPUANO ? res_fixed_words<ISG_RNG_PARISI_RAPUANO>() : 0;
    P.smem = sizeof(uint32_t) * (size_t)(2 * P.cw * (pairs ? pairs : 1) + fixed + pieces * stream);
    return P;
}

static void fill_args(isg_sim* h, const ResidentLayout& P, ResidentArgs& A) {
    A.a = make_flip_args(h, 0);
    A.npass = 0;
    A.parts = P.parts;
    A.rpb = P.rpb;
    A.ncta = P.ncta;
    A.cw = P.cw;
    auto magic = [](uint64_t d) { return (uint32_t)(((1ull << 32) + d - 1) / d); };
    A.mW = magic((uint64_t)h->W);
    A.mL = magic((uint64_t)h->L);
    A.mR = magic((uint64_t)h->R);
    A.done = nullptr;
    A.err = nullptr;
    A.stall = 0;
    A.usum = nullptr;
    A.jumps = nullptr;
    A.rng_in = A.a.rng;
    A.rng_out = nullptr;
    A.lv = nullptr;
    A.lv_pass = 0;
}

// Whether `blocks` blocks of fn with `smem` bytes each can all be resident.
template <class Fn>
static bool all_fit(Fn fn, int threads, size_t smem, int64_t blocks, int sms) {
    if (smem > 227 * 1024) return false;
    if (smem > 48 * 1024 &&
        cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    int occ = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, fn, threads, smem) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return (int64_t)occ * sms >= blocks;
}

static bool cooperative_device() {
    int coop = 0;
    return cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, current_device()) == cudaSuccess && coop;
}

template <class Fn, class... Args>
static cudaError_t launch_cooperative(Fn fn, int grid, int threads, size_t smem, cudaStream_t s, const Args&... args) {
    cudaLaunchConfig_t lc = {};
    lc.gridDim = dim3((unsigned)grid);
    lc.blockDim = dim3((unsigned)threads);
    lc.dynamicSmemBytes = smem;
    lc.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
    lc.attrs = at;
    lc.numAttrs = 1;
    return cudaLaunchKernelEx(&lc, fn, args...);
}

struct ResidentPlan {
    ResidentLayout lay;
    ResidentLayout apart;      // of minstd_pass_kernel
    bool one_apart = false;    // calls of one sweep are two of its launches
    int pairs = 0, minb = 4, threads = 0;
    PrJumps jumps;
};

template <typename Word, int KIND, int PAIRS, int MINB>
static auto resident_fn() {
    if constexpr (KIND == ISG_RNG_PARISI_RAPUANO) return resident_kernel<Word, KIND, PAIRS, MINB, PrJumps>;
    else return resident_kernel<Word, KIND, PAIRS, MINB, NoJumps>;
}

template <int KIND, int PAIRS, int MINB>
static auto resident_set_fn() {
    if constexpr (KIND == ISG_RNG_PARISI_RAPUANO) return resident_set_kernel<KIND, PAIRS, MINB, PrTo>;
    else return resident_set_kernel<KIND, PAIRS, MINB, NoJumps>;
}

template <typename Word, int KIND, int PAIRS, int MINB>
static bool plan_for(const isg_sim* h, int sms, ResidentPlan& P) {
    P.pairs = PAIRS;
    P.minb = MINB;
    P.threads = PAIRS ? 64 * PAIRS : kResThreads;
    P.lay = layout_of(h, PAIRS, (int64_t)sms * MINB);
    return all_fit(resident_fn<Word, KIND, PAIRS, MINB>(), P.threads, P.lay.smem, P.lay.ncta, sms);
}

// f(PAIRS, MINB) of the MT19937 kernels
template <class F>
static auto with_pairs(int pairs, int minb, F&& f) {
    using std::integral_constant;
    if (pairs == 1 && minb <= 10) return f(integral_constant<int, 1>{}, integral_constant<int, 10>{});
    if (pairs == 1) return f(integral_constant<int, 1>{}, integral_constant<int, 14>{});
    if (pairs == 4 && minb <= 2) return f(integral_constant<int, 4>{}, integral_constant<int, 2>{});
    if (pairs == 4 && minb <= 3) return f(integral_constant<int, 4>{}, integral_constant<int, 3>{});
    if (pairs == 4) return f(integral_constant<int, 4>{}, integral_constant<int, 4>{});
    return f(integral_constant<int, 0>{}, integral_constant<int, 4>{});
}

template <typename Word, int KIND>
static bool make_plan(const isg_sim* h, int sms, ResidentPlan& best) {
    bool found = false;
    if constexpr (KIND == ISG_RNG_MT19937) {
        const int per = (int)((h->S + sms - 1) / sms);  // streams of the fullest SM
        // up to three: seven warps a stream (L = 192, per = 2: 9.4 us a pass against
        // 13.7 with pairs; L = 256, per = 4: 19.7 against 13.6).  Then blocks of
        // one pair, or of four where rounding the fullest SM up to whole blocks
        // adds at most one stream (L = 384, per = 12: 36.7 us against 41.0 with
        // blocks of one; L = 352, per = 9: 38.3 against 32.4).  Against a launch per
        // pass, calls of 32 sweeps: L = 300 41.9 -> 20.1, L = 352 45.0 -> 33.1,
        // L = 400 62.2 -> 53.5
        const int pairs = per <= 3 ? 0 : per > 6 && (per + 1) % 4 <= 1 ? 4 : 1;
        found = with_pairs(pairs, pairs == 1 ? per : (per + 3) / 4, [&](auto p, auto m) {
            return plan_for<Word, KIND, decltype(p)::value, decltype(m)::value>(h, sms, best);
        });
    } else {
        found = plan_for<Word, KIND, 0, 4>(h, sms, best);
    }
    if (found && KIND == ISG_RNG_PARISI_RAPUANO) {
        best.jumps.to = pr_to();
        pr_pass(h, best.jumps.pass);
    }
    if (KIND == ISG_RNG_MINSTD) {
        // Calls of one sweep: a cooperative launch costs about 7 us beyond its passes,
        // two ordinary ones that overlap (programmatic dependent launch) about 2.  us
        // per call, one behind the other, resident -> apart: L = 128 10.4 -> 8.5, 150
        // 14.4 -> 11.2, 192 16.2 -> 12.3, 212 17.3 -> 12.7, 256 20.9 -> 17.7, 280 28.9 ->
        // 25.4; where each call is waited for 24.1 -> 22.9, 27.5 -> 25.4, .., 34.1 -> 34.0.
        // Not below a quarter of a stream an SM (L = 64: 1 us less, waited for 0.3 more),
        // nor from five on (L = 320 34.9 -> 33.0, waited for 47.9 -> 48.7), nor for two
        // sweeps (L = 188 22.6 -> 23.8, waited for 36.4 -> 40.0).  Blocks: two an SM
        // (L = 212 / 276: 12.7 / 24.6, four 13.1 / 26.1), four where two of even shares
        // come out half a stream too large (L = 236 17.0 -> 15.9); even shares where whole
        // parts of streams leave an SM with twice another's (L = 188 13.0 -> 12.0).
        const int64_t S20 = 20 * h->S / sms;  // streams per SM, in twentieths
        best.one_apart = S20 >= 5 && S20 < 100;
        best.apart = layout_of(h, 0, (int64_t)sms * (S20 >= 44 && S20 < 68 ? 4 : 2),
                               (S20 >= 17 && S20 < 32) || (S20 >= 44 && S20 < 68));
    }
    return found;
}

// The layout of h's resident launches, made on first use and kept (NULL: none).
static const ResidentPlan* resident_plan(isg_sim* h) {
    if (h->res_plan || h->res_none) return (const ResidentPlan*)h->res_plan;
    ResidentPlan* P = new (std::nothrow) ResidentPlan();
    const int sms = sm_count();
    const bool ok = P && cooperative_device() && with_kind(h->kind, [&](auto kind) {
                        constexpr int K = decltype(kind)::value;
                        return h->wbits == 64 ? make_plan<uint64_t, K>(h, sms, *P) : make_plan<uint32_t, K>(h, sms, *P);
                    });
    if (!ok) {
        delete P;
        h->res_none = true;
        return nullptr;
    }
    h->res_plan = P;
    return P;
}

void free_resident_plan(void* p) { delete (ResidentPlan*)p; }

// Streams per SM below which the resident launches are the better way: 16 for
// MT19937 and MINSTD (all sizes whose blocks fit on the GPU; L = 428: 74.1 ->
// 56.8 and 42.5 -> 31.4 us per pass), 8 for Parisi-Rapuano, whose calls of one
// sweep pay for the jumps to the pieces' starts (L = 320: 94.5 -> 82 us, at
// L = 428 it would be 122 -> 147 us).
bool resident_size(const isg_sim* h) {
    return h->S < (h->kind == ISG_RNG_PARISI_RAPUANO ? 8 : 16) * (int64_t)sm_count();
}

// MT19937: at least one whole stream a block; else the blocks of plan_for.
size_t resident_count_bytes(const isg_sim* h) {
    const int64_t blocks = h->kind == ISG_RNG_MT19937 ? h->S : layout_of(h, 0, (int64_t)sm_count() * 4).ncta;
    return (size_t)blocks * sizeof(unsigned long long);
}

static bool capturing(cudaStream_t s) {
    cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(s, &st) == cudaSuccess) return st != cudaStreamCaptureStatusNone;
    cudaGetLastError();
    return true;
}

bool sweeps_resident(isg_sim* h) { return resident_size(h) && h->done && resident_plan(h) != nullptr; }

template <typename Word, int KIND>
static cudaError_t launch_plan(const ResidentPlan* P, const ResidentArgs& A, cudaStream_t s) {
    const StreamConst K = stream_const();
    auto go = [&](auto fn, const auto& J) {
        return launch_cooperative(fn, P->lay.ncta, P->threads, P->lay.smem, s, A, K, J);
    };
    if constexpr (KIND == ISG_RNG_MT19937)
        return with_pairs(P->pairs, P->minb, [&](auto p, auto m) {
            return go(resident_fn<Word, KIND, decltype(p)::value, decltype(m)::value>(), NoJumps{});
        });
    else if constexpr (KIND == ISG_RNG_PARISI_RAPUANO)
        return go(resident_fn<Word, KIND, 0, 4>(), P->jumps);
    else
        return go(resident_fn<Word, KIND, 0, 4>(), NoJumps{});
}

// One sweep of a MINSTD lattice as a launch a pass (programmatic dependent launch).
// The red pass leaves the states in rng_pos, which MINSTD has no other use for, the
// blue one puts them back.
static cudaError_t launch_minstd_apart(isg_sim* h, const ResidentLayout& lay, cudaStream_t s,
                                       unsigned long long* usum) {
    ResidentArgs A;
    fill_args(h, lay, A);
    A.err = (unsigned long long*)(h->scal + 5);
    A.npass = 1;
    const StreamConst K = stream_const();
    cudaLaunchConfig_t lc = {};
    lc.gridDim = dim3((unsigned)lay.ncta);
    lc.blockDim = dim3(kResThreads);
    lc.dynamicSmemBytes = lay.smem;
    lc.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    lc.attrs = at;
    lc.numAttrs = 1;
    for (int c = 0; c < 2; ++c) {
        A.a.c = c;
        A.rng_in = c ? h->rng_pos : h->rng;
        A.rng_out = c ? h->rng : h->rng_pos;
        A.usum = c ? nullptr : usum;
        const cudaError_t e = h->wbits == 64 ? cudaLaunchKernelEx(&lc, minstd_pass_kernel<uint64_t>, A, K)
                                             : cudaLaunchKernelEx(&lc, minstd_pass_kernel<uint32_t>, A, K);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

cudaError_t launch_resident(isg_sim* h, int64_t n, cudaStream_t s, unsigned long long* usum) {
    const ResidentPlan* P = resident_plan(h);
    if (!P) return cudaErrorNotSupported;
    if (n == 1 && P->one_apart && !h->res_stall) return launch_minstd_apart(h, P->apart, s, usum);
    ResidentArgs A;
    fill_args(h, P->lay, A);
    A.done = h->done;
    A.err = (unsigned long long*)(h->scal + 5);
    for (int64_t left = 2 * n; left > 0;) {
        const int64_t np = std::min<int64_t>(left, kResidentPasses);
        A.npass = (int)np;
        A.stall = h->res_stall ? 1ull : 0ull;
        A.usum = usum;
        usum = nullptr;
        const cudaError_t e = with_kind(h->kind, [&](auto kind) {
            constexpr int K = decltype(kind)::value;
            return h->wbits == 64 ? launch_plan<uint64_t, K>(P, A, s) : launch_plan<uint32_t, K>(P, A, s);
        });
        if (e != cudaSuccess) return e;
        h->res_stall = false;
        left -= np;
    }
    return cudaSuccess;
}

// ------------------------------------------------------ several lattices ---
// f(PAIRS, MINB) of the MT19937 kernels of several lattices
template <class F>
static auto with_set_pairs(int pairs, int minb, F&& f) {
    using std::integral_constant;
    if (pairs == 1 && minb <= 4) return f(integral_constant<int, 1>{}, integral_constant<int, 4>{});
    if (pairs == 1 && minb <= 10) return f(integral_constant<int, 1>{}, integral_constant<int, 10>{});
    if (pairs == 1) return f(integral_constant<int, 1>{}, integral_constant<int, 14>{});
    return f(integral_constant<int, 0>{}, integral_constant<int, 4>{});
}

template <int KIND, class F>
static auto with_set_fn(const ResidentSet& R, F&& f) {
    if constexpr (KIND == ISG_RNG_MT19937)
        return with_set_pairs(R.pairs, R.minb, [&](auto p, auto m) {
            return f(resident_set_fn<KIND, decltype(p)::value, decltype(m)::value>());
        });
    else
        return f(resident_set_fn<KIND, 0, 4>());
}

static void set_free(ResidentSet& R) {
    if (R.owner) dev_free(R.owner, R.d_mem);
    else cudaFree(R.d_mem);
    R.d_mem = nullptr;
    R.cap = 0;
}

void ResidentSet::clear() {
    set_free(*this);
    nblocks = 0;
}

bool ResidentSet::plan(int kind_, const std::vector<isg_sim*>& sims, unsigned long long* err) {
    nblocks = 0;
    most = 0;
    kind = kind_;
    const int sms = sm_count();
    if (sims.empty() || !cooperative_device()) return false;
    int64_t streams = 0, rows = 0;
    for (const isg_sim* h : sims) {
        if (h->wbits != 64 || h->kind != kind) return false;
        streams += h->S;
        rows += h->rows * h->W;
    }
    // Streams per SM up to which one launch is the better way for all lattices
    // together: MT19937 14 (one pair of warps each; more do not fit; against a launch
    // per pass, 64 sweeps of 40 x 2, 60 x 2, 120 x 2 lattices of L = 64, 5, 7 and 13
    // streams per SM, 5.72 -> 2.59, 5.92 -> 3.26, 8.02 -> 5.44 ms; in a server, beside
    // the other kinds' launches, 4: with 14, 40 draws of 24 jobs took 13 % less in the
    // mean, but seven of them 3 to 18 % more), Parisi-Rapuano
    // 12, MINSTD 48 where the other way is a launch per pass (a server's quanta), 28
    // where it is the group passes (batches).  64 sweeps of batches of n samples of
    // mixed size, resident / launch per pass / group passes, ms: MINSTD n = 32
    // 5.3 / - / 7.1, 48 9.2 / - / 8.3, 64 11.0 / 14.0 / 9.0, 128 24.4 / 20.7 / 15.3;
    // Parisi-Rapuano n = 8 4.4 / - / 6.7, 16 7.6 / - / 7.3
    const int per = (int)((streams + sms - 1) / sms);
    pairs = 0;
    minb = 4;
    int64_t share = 0;  // MINSTD, Parisi-Rapuano: words of a block
    if (kind == ISG_RNG_MT19937) {
        if (per > mt_most) return false;
        pairs = per <= 3 ? 0 : 1;
        minb = pairs ? per : 4;
    } else {
        if (per > (kind == ISG_RNG_PARISI_RAPUANO ? 12 : minstd_most)) return false;
        const int64_t cap_blocks = (int64_t)sms * 4;
        if ((int64_t)sims.size() > cap_blocks) return false;
        share = std::max<int64_t>(64, (rows + cap_blocks - 1) / cap_blocks);
        for (;;) {  // the smallest share whose blocks fit
            int64_t n = 0;
            for (const isg_sim* h : sims)
                n += layout_of(h, 0, std::max<int64_t>(1, h->rows * h->W / share)).ncta;
            if (n <= cap_blocks) break;
            if (share > rows) return false;
            share += (share + 15) / 16;
        }
    }
    threads = pairs ? 64 * pairs : kResThreads;
    std::vector<ResidentArgs> tab(sims.size());
    std::vector<PrPass> jumps;
    std::vector<int2> blocks;
    std::vector<int> order(sims.size()), first(sims.size());
    smem = 0;
    int64_t n = 0;
    for (size_t i = 0; i < sims.size(); ++i) {
        isg_sim* h = sims[i];
        const ResidentLayout P = layout_of(h, pairs, pairs || kind == ISG_RNG_MT19937
                                                         ? 1 : std::max<int64_t>(1, h->rows * h->W / share));
        fill_args(h, P, tab[i]);
        smem = std::max(smem, P.smem);
        first[i] = (int)n;
        n += P.ncta;
        for (int b = 0; b < P.ncta; ++b) blocks.push_back(make_int2((int)i, b));
        if (kind == ISG_RNG_PARISI_RAPUANO) {
            size_t q = 0;  // lattices of one size share theirs
            while (q < i && sims[q]->L != h->L) ++q;
            order[i] = q < i ? order[q] : (int)jumps.size();
            if (q == i) {
                jumps.emplace_back();
                pr_pass(h, jumps.back());
            }
        }
    }
    const bool fits = with_kind(kind, [&](auto kc) {
        return with_set_fn<decltype(kc)::value>(*this, [&](auto fn) { return all_fit(fn, threads, smem, n, sms); });
    });
    if (!fits) return false;
    // one device allocation: table, blocks, jumps, counts
    auto up = [](size_t v) { return (v + 255) / 256 * 256; };
    const size_t o_blocks = up(tab.size() * sizeof tab[0]), o_jumps = o_blocks + up(blocks.size() * sizeof blocks[0]);
    const size_t o_done = o_jumps + up(jumps.size() * sizeof(PrPass));
    const size_t bytes = o_done + up((size_t)n * sizeof(unsigned long long));
    if (bytes > cap) {
        set_free(*this);
        if (owner) d_mem = dev_alloc(owner, 2 * bytes);
        else if (cudaMalloc(&d_mem, 2 * bytes) != cudaSuccess) {
            cudaGetLastError();
            d_mem = nullptr;
        }
        if (!d_mem) return false;
        cap = 2 * bytes;
    }
    char* m = (char*)d_mem;
    for (size_t i = 0; i < tab.size(); ++i) {
        tab[i].done = (unsigned long long*)(m + o_done) + first[i];
        tab[i].err = err;
        if (kind == ISG_RNG_PARISI_RAPUANO) tab[i].jumps = (const PrPass*)(m + o_jumps) + order[i];
    }
    host.assign(o_done, 0);
    memcpy(host.data(), tab.data(), tab.size() * sizeof tab[0]);
    memcpy(host.data() + o_blocks, blocks.data(), blocks.size() * sizeof blocks[0]);
    if (!jumps.empty()) memcpy(host.data() + o_jumps, jumps.data(), jumps.size() * sizeof(PrPass));
    off_blocks = o_blocks;
    off_done = o_done;
    nsims = (int)sims.size();
    nblocks = (int)n;
    uploaded = false;
    return true;
}

void ResidentSet::set_passes(int i, int npass) {
    ((ResidentArgs*)host.data())[i].npass = npass;
    most = std::max(most, npass);
}

void ResidentSet::set_stall(int i) {
    ((ResidentArgs*)host.data())[i].stall = 1ull;
    uploaded = false;
}

void ResidentSet::reset() {
    for (int i = 0; i < nsims && nblocks; ++i) ((ResidentArgs*)host.data())[i].stall = 0ull;
    uploaded = false;
}

cudaError_t ResidentSet::launch(int npass, cudaStream_t s) {
    if (!uploaded) {
        cudaError_t e = cudaMemcpyAsync(d_mem, host.data(), host.size(), cudaMemcpyHostToDevice, s);
        if (e == cudaSuccess)
            e = cudaMemsetAsync((char*)d_mem + off_done, 0, (size_t)nblocks * sizeof(unsigned long long), s);
        if (e != cudaSuccess) return e;
        uploaded = !capturing(s);  // a captured upload runs when the graph does
    }
    const ResidentArgs* tab = (const ResidentArgs*)d_mem;
    const int2* blocks = (const int2*)((const char*)d_mem + off_blocks);
    const StreamConst K = stream_const();
    const int all = npass > 0 ? npass : most;
    cudaError_t e = cudaSuccess;
    for (int first = 0; first < all && e == cudaSuccess; first += kResidentPasses)
        e = with_kind(kind, [&](auto kc) {
            constexpr int KIND = decltype(kc)::value;
            return with_set_fn<KIND>(*this, [&](auto fn) {
                if constexpr (KIND == ISG_RNG_PARISI_RAPUANO)
                    return launch_cooperative(fn, nblocks, threads, smem, s, tab, blocks, npass, first, K,
                                              pr_to());
                else
                    return launch_cooperative(fn, nblocks, threads, smem, s, tab, blocks, npass, first, K, NoJumps{});
            });
        });
    return e;
}

// ---------------------------------------------------------- levels alone ---
// MINSTD and Parisi-Rapuano that write out levels only: the states of the parts
// of a stream are all read from where its first part's block stores them back,
// so the launch reads a copy of them.
bool LevelsPlan::make(const isg_sim& g) {
    const int sms = sm_count();
    kind = g.kind;
    const bool mt = kind == ISG_RNG_MT19937;
    const int per = (int)((g.S + sms - 1) / sms);
    bytes = mt && per > 3;  // a pair of warps a stream; else seven (or 256 threads a part)
    ResidentLayout P;
    P.rpb = (int)g.R;
    if (!mt) {  // parts of at least 1024 draws, four blocks per SM
        const int64_t least = (1024 + g.half - 1) / g.half;
        const int64_t parts_ = std::max<int64_t>(1, std::min((g.R + least - 1) / least, (int64_t)sms * 4 / g.S));
        P.rpb = (int)((g.R + parts_ - 1) / parts_);
    }
    P.parts = (int)((g.R + P.rpb - 1) / P.rpb);
    P.ncta = (int)g.S * P.parts;
    const int D = P.rpb * g.half;
    P.cw = (D / 32 + 20 + 3) / 4 * 4;
    const int stream = mt ? res_stream_words<ISG_RNG_MT19937>()
                          : (kind == ISG_RNG_MINSTD ? res_stream_words<ISG_RNG_MINSTD>()
                                                    : res_stream_words<ISG_RNG_PARISI_RAPUANO>());
    P.smem = sizeof(uint32_t) * (size_t)(2 * P.cw + stream +
                                         (kind == ISG_RNG_PARISI_RAPUANO ? res_fixed_words<ISG_RNG_PARISI_RAPUANO>() : 0));
    if (P.smem > 48 * 1024) return false;
    parts = P.parts;
    rpb = P.rpb;
    nblocks = P.ncta;
    cw = P.cw;
    smem = P.smem;
    pass_words = (size_t)nblocks * 2 * cw;
    state_bytes = mt ? 0 : (size_t)g.S * rng_state_words(kind) * 4;
    if (kind == ISG_RNG_PARISI_RAPUANO) {
        PrJumps* J = new (std::nothrow) PrJumps();
        if (!J) return false;
        J->to = pr_to();
        pr_pass(&g, J->pass);
        jumps = J;
    }
    return true;
}

void LevelsPlan::clear() {
    delete (PrJumps*)jumps;
    jumps = nullptr;
}

cudaError_t LevelsPlan::launch(const FlipArgs& gen, uint32_t* rng_copy, uint32_t* lv, int npass, cudaStream_t s) const {
    ResidentArgs A;
    memset(&A, 0, sizeof A);
    A.a = gen;
    A.npass = npass;
    A.parts = parts;
    A.rpb = rpb;
    A.ncta = nblocks;
    A.cw = cw;
    A.lv = lv;
    A.lv_pass = (int64_t)pass_words;
    A.rng_in = gen.rng;
    if (state_bytes) {
        const cudaError_t e = cudaMemcpyAsync(rng_copy, gen.rng, state_bytes, cudaMemcpyDeviceToDevice, s);
        if (e != cudaSuccess) return e;
        A.rng_in = rng_copy;
    }
    const StreamConst K = stream_const();
    if (kind == ISG_RNG_MT19937) {
        if (bytes) levels_kernel<ISG_RNG_MT19937, 1, NoJumps><<<nblocks, 64, smem, s>>>(A, K, NoJumps{});
        else levels_kernel<ISG_RNG_MT19937, 0, NoJumps><<<nblocks, kResThreads, smem, s>>>(A, K, NoJumps{});
    } else if (kind == ISG_RNG_PARISI_RAPUANO) {
        levels_kernel<ISG_RNG_PARISI_RAPUANO, 0, PrJumps><<<nblocks, kResThreads, smem, s>>>(A, K, *(const PrJumps*)jumps);
    } else {
        levels_kernel<ISG_RNG_MINSTD, 0, NoJumps><<<nblocks, kResThreads, smem, s>>>(A, K, NoJumps{});
    }
    return cudaGetLastError();
}

}  // namespace isg
