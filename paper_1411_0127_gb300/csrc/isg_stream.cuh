// isg_stream.cuh -- one warp's colour pass over one RNG stream, shared by the
// single-lattice kernel (isg_flip_fast.cu) and the batched engine (isg_batch.cu),
// and the word updates and draw steps that the resident launches
// (isg_resident.cu) use as well.
//
// A stream owns R consecutive rows r = y + L*z of a lattice.  The warp walks
// them in groups of G = 32 / W rows (W words per row and colour), one word of
// the group per lane:
//   1. draw phase: the group's draws are produced 128 at a time in stream order
//      (row by row, ascending x) and compared with the three integer thresholds
//      thr1 > thr2 > thr3 (Sec. 4: R < Rmax exp(-beta dE)).  Because the three
//      comparisons are nested, a draw's outcome is a level 0..3 (how many
//      thresholds it is below): "lo" = level odd, "hi" = level >= 2.  They are
//      left in shared memory: by MINSTD and Parisi-Rapuano as two bit streams,
//      from two ballots per 32 draws; by MT19937, whose lanes make four
//      consecutive draws each, as a byte a lane (lo bits in the low nibble, hi
//      bits in the high one);
//   2. logic phase: each lane loads its word of S_c, its forward couplings and
//      the other colour's neighbour words, counts unsatisfied bonds with a
//      bit-sliced adder, cuts its window out of the levels
//      (d < thr1 = lo | hi, d < thr2 = hi, d < thr3 = lo & hi), forms the flip
//      mask, XORs it into S_c and sums dE = 12 - 4u.
//
// Generators (Sec. 3):
//   * MT19937 keeps its words in a linear window of shared memory: B[j] holds
//     x_{base + j}, x_{k+624} is appended at B[k - base + 624], and when the
//     free slots run out the 624 live words move back to the front; the reads
//     x_k, x_{k+1}, x_{k+397} are fixed offsets from one index with no
//     wrap-around arithmetic.  Its shifts run as multiplies (MtMul) on the FMA
//     pipe;
//   * MINSTD keeps two lanes' worth of states (positions +1..+32 and +33..+64)
//     and compares the state x with ceil(thr / 2) (d = 2x < thr <=> x <
//     ceil(thr / 2));
//   * Parisi-Rapuano keeps its 64-word window in two registers per lane
//     (pr_warp_step in isg_common.cuh): no shared memory.
#pragma once

#include "isg_common.cuh"

namespace isg {

// Multipliers that turn the generator's shifts into integer multiplies:
// v >> k == umulhi(v, 2^(32-k)) and v << k == v * 2^k (mod 2^32), exactly.
// They arrive as kernel arguments so that the compiler cannot fold them back
// into shift instructions: the multiplies run on the FMA pipe, leaving only the
// XORs on the (half-rate) logic pipe.
struct MtMul {
    uint32_t hi31;  // 2^31: >> 1
    uint32_t hi21;  // 2^21: >> 11
    uint32_t hi14;  // 2^14: >> 18
    uint32_t lo7;   // 2^7:  << 7
    uint32_t lo15;  // 2^15: << 15
    uint32_t two;   // 2: a doubling as a multiply-add (push_compare)
};

// Per-launch generator constants.
struct StreamConst {
    MtMul mul;
    uint32_t a32;   // 16807^32 mod (2^31 - 1)
    uint32_t a64;   // 16807^64 mod (2^31 - 1)
};

inline StreamConst stream_const() {
    const MinstdTable t = minstd_table();
    StreamConst k;
    k.mul.hi31 = 1u << 31;
    k.mul.hi21 = 1u << 21;
    k.mul.hi14 = 1u << 14;
    k.mul.lo7 = 1u << 7;
    k.mul.lo15 = 1u << 15;
    k.mul.two = 2u;
    k.a32 = t.pow[32];
    k.a64 = minstd_mulmod(t.pow[32], t.pow[32]);
    return k;
}

// Shared-memory words of one warp's MT19937 window with `slack` free slots.
constexpr int mt_window(int slack) { return kMtN + slack; }

// MT19937 twist of one word: x_{k+624} from x_k, x_{k+1}, x_{k+397}.  y and
// x_{k+1} share their low bit, so the odd test is y - 2 (y >> 1) = y & 1, one
// multiply-add on the shift y >> 1 that the twist needs anyway (testing the
// low bit of x_{k+1} by its own shift cost one more FMA-pipe instruction per
// draw: L = 1024 MT19937 1.169 -> 1.101 ps per attempt without it).
__device__ __forceinline__ uint32_t mt_twist(uint32_t a, uint32_t b, uint32_t m, const MtMul& k) {
    const uint32_t y = (a & 0x80000000u) | (b & 0x7FFFFFFFu);
    const uint32_t ys = __umulhi(y, k.hi31);
    const uint32_t odd = y - 2u * ys;
    return m ^ ys ^ (odd * 0x9908B0DFu);
}

// MT19937 tempering with the shifts done as multiplies (see MtMul).
__device__ __forceinline__ uint32_t mt_temper_mul(uint32_t v, const MtMul& k) {
    v ^= __umulhi(v, k.hi21);
    v ^= (v * k.lo7) & 0x9D2C5680u;
    v ^= (v * k.lo15) & 0xEFC60000u;
    v ^= __umulhi(v, k.hi14);
    return v;
}

// The three compare values of a pass, held in registers: the batched engine
// reads its FlipArgs from global memory, where the compiler could not keep them
// across the shared-memory stores of the draw loop.
struct Cmp {
    uint32_t c1, c2, c3;
};

__device__ __forceinline__ Cmp cmp_of(const FlipArgs& a) { return Cmp{a.cmp1, a.cmp2, a.cmp3}; }

// Four consecutive draws a thread: the quads x_k .. x_{k+3} and x_{k+396} ..
// x_{k+399} come as 16-byte loads and the words after them, x_{k+4} and
// x_{k+400}, as single ones, so 128 draws take four loads and a store of shared
// memory instead of sixteen.  `a`, `m` hold the quads, `an`, `mn` the words after.
__device__ __forceinline__ void mt_twist4(const uint4& a, uint32_t an, const uint4& m, uint32_t mn, uint32_t (&v)[4],
                                          const MtMul& k) {
    v[0] = mt_twist(a.x, a.y, m.y, k);
    v[1] = mt_twist(a.y, a.z, m.z, k);
    v[2] = mt_twist(a.z, a.w, m.w, k);
    v[3] = mt_twist(a.w, an, mn, k);
}

// Compare values of the four-draw form.  The last tempering step, d = z ^ (z >> 18),
// leaves the upper 18 bits alone, so d < c1 is z < C = (c1 with its low 14 bits
// cleared) unless z lies in [C, C + 2^14); and if z > (c2 | 0x3FFF), d > c2.  With
// t = z - C (mod 2^32), a warp none of whose z and t are at most c2 | 0x3FFF has
// no such draw and none below c2 >= c3, and needs neither the last step nor the
// other comparisons.  z - C is an addition whose carry is the comparison.
struct Cmp4 {
    uint32_t negC;   // -C mod 2^32
    uint32_t rare;   // c2 | 0x3FFF
    uint32_t mask;   // 15, or 0 if C = 0 (then every draw that is not rare is not below c1)
};

__device__ __forceinline__ Cmp4 cmp4_of(const Cmp& c) {
    const uint32_t C = c.c1 & ~0x3FFFu;
    return Cmp4{0u - C, c.c2 | 0x3FFFu, C ? 15u : 0u};
}

// acc = 2 acc + (z >= C), returns t = z - C mod 2^32: an addition whose carry goes
// into a multiply-add (the FMA pipe has room).
__device__ __forceinline__ uint32_t push_compare(uint32_t& acc, uint32_t z, uint32_t negC, const MtMul& k) {
    uint32_t t;
    asm("add.cc.u32 %0, %2, %3;\n\tmadc.lo.u32 %1, %1, %4, 0;" : "=&r"(t), "+r"(acc) : "r"(z), "r"(negC), "r"(k.two));
    return t;
}

__device__ __forceinline__ uint32_t min3(uint32_t a, uint32_t b, uint32_t c) { return min(min(a, b), c); }

// Level byte (see take_levels) of a lane's four consecutive draws, from the raw
// words v, in two halves: the tempering and the comparisons of the common case,
// then the warp's vote on whether it is one.  Warp-wide.
struct LevelHalf {
    uint32_t z[4], byte, low;
};

__device__ __forceinline__ LevelHalf mt_level_begin(const uint32_t (&v)[4], const Cmp4& c4, const MtMul& k) {
    LevelHalf h;
    uint32_t t[4], acc = 0;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        uint32_t z = v[i] ^ __umulhi(v[i], k.hi21);
        z ^= (z * k.lo7) & 0x9D2C5680u;
        h.z[i] = z ^ ((z * k.lo15) & 0xEFC60000u);
    }
#pragma unroll
    for (int i = 3; i >= 0; --i) t[i] = push_compare(acc, h.z[i], c4.negC, k);
    h.low = min3(min3(h.z[0], h.z[1], h.z[2]), h.z[3], min(t[0], min3(t[1], t[2], t[3])));
    h.byte = ~acc & c4.mask;
    return h;
}

// REDUX: the vote as a minimum over the warp, whose result is in a uniform
// register; faster in the multi-pass launches of one lattice (L = 1024 1.015 ->
// 0.994 ps per attempt, L = 640 1.088 -> 1.070), slower in the other kernels (the
// batch's pass launches 120.2 -> 120.9 ms, L = 512 1.219 -> 1.231 ps).
template <bool REDUX = false>
__device__ __forceinline__ uint32_t mt_level_finish(const LevelHalf& h, const Cmp& c, const Cmp4& c4) {
    uint32_t byte = h.byte;
    if (REDUX ? __reduce_min_sync(kFull, h.low) <= c4.rare : __any_sync(kFull, h.low <= c4.rare)) {
        byte = 0;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const uint32_t d = h.z[i] ^ (h.z[i] >> 18);
            const uint32_t hi = d < c.c2 ? 1u : 0u, lo = (d < c.c1 ? 1u : 0u) ^ hi ^ (d < c.c3 ? 1u : 0u);
            byte |= (lo << i) | (hi << (4 + i));
        }
    }
    return byte;
}

// Make room for `need` more words: if the window is full, move the 624 live
// words B[iA .. iA+623] to the front (all read before any is written).
template <int SLACK>
__device__ __forceinline__ void mt_make_room(uint32_t* B, int& iA, int need, int lane) {
    if (iA + kMtN + need <= mt_window(SLACK)) return;
    __syncwarp();
    if ((iA & 3) == 0) {  // 16-byte aligned four-word moves
        constexpr int n4 = kMtN / 4, kPer = (n4 + 31) / 32;
        uint4 v[kPer];
#pragma unroll
        for (int q = 0; q < kPer; ++q)
            if (lane + 32 * q < n4) v[q] = *(const uint4*)(B + iA + 4 * (lane + 32 * q));
        __syncwarp();
#pragma unroll
        for (int q = 0; q < kPer; ++q)
            if (lane + 32 * q < n4) *(uint4*)(B + 4 * (lane + 32 * q)) = v[q];
        iA = 0;
    } else {
        uint32_t v[20];
#pragma unroll
        for (int q = 0; q < 20; ++q) v[q] = (lane + 32 * q < kMtN) ? B[iA + lane + 32 * q] : 0u;
        __syncwarp();
#pragma unroll
        for (int q = 0; q < 20; ++q)
            if (lane + 32 * q < kMtN) B[lane + 32 * q] = v[q];
        iA = 0;
    }
    __syncwarp();
}

// 128 draws, four consecutive ones a lane (iA a multiple of 4): the raw words
// x_{k+624+4l} .. +3, appended to the window.  The reads (up to k + 524) and the
// writes (from k + 624) of a step never meet, so the warp barrier after the
// writes is the only one.  The two single words cost four shared-memory
// wavefronts each (lanes l and l + 8 meet in a bank); taken from the next lane by
// shuffles, with a load for lane 31, they were slower (L = 1024 1.024 - 1.066
// against 1.011 ps).
__device__ __forceinline__ void mt_quad4(uint32_t* B, int& iA, uint32_t (&v)[4], const MtMul& k, int lane) {
    const uint32_t* q = B + iA + 4 * lane;
    const uint4 a = *(const uint4*)q;
    const uint4 m = *(const uint4*)(q + kMtM - 1);
    const uint32_t an = q[4], mn = q[kMtM + 3];
    mt_twist4(a, an, m, mn, v, k);
    *(uint4*)(B + iA + 4 * lane + kMtN) = make_uint4(v[0], v[1], v[2], v[3]);
    __syncwarp();
    iA += 128;
}

// Four 32-draw blocks (128 draws) at once.  Block j reads x_{k+32j+l+397},
// which was appended 227 - 32j - l >= 100 draws before this step; the step's
// reads (indices up to k + 524) and writes (from k + 624) never meet, so the
// one warp barrier after the writes, which orders them before the next step's
// reads, is the only one (a second one between the reads and the writes cost
// 0.7 % at L = 1024).
template <int SLACK, bool ROOM = true>
__device__ __forceinline__ void mt_quad(uint32_t* B, int& iA, uint32_t d[4], const MtMul& k, int lane) {
    if (ROOM) mt_make_room<SLACK>(B, iA, 128, lane);
    uint32_t a[4], b[4], m[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const int i = iA + 32 * j + lane;
        a[j] = B[i];
        b[j] = B[i + 1];
        m[j] = B[i + kMtM];
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const uint32_t v = mt_twist(a[j], b[j], m[j], k);
        B[iA + 32 * j + lane + kMtN] = v;
        d[j] = v;
    }
    __syncwarp();
    iA += 128;
#pragma unroll
    for (int j = 0; j < 4; ++j) d[j] = mt_temper_mul(d[j], k);
}

// One block of up to 32 draws (tail of a row group); lanes >= nvalid consume
// nothing.  Reads reach k + 428 and writes start at k + 624: one barrier, after
// the writes.
template <int SLACK>
__device__ __forceinline__ uint32_t mt_single(uint32_t* B, int& iA, int lane, int nvalid, const MtMul& k) {
    mt_make_room<SLACK>(B, iA, 32, lane);
    const int i = iA + lane;
    const uint32_t a = B[i], b = B[i + 1], m = B[i + kMtM];
    const uint32_t v = mt_twist(a, b, m, k);
    if (lane < nvalid) B[i + kMtN] = v;
    __syncwarp();
    iA += nvalid;
    return mt_temper_mul(v, k);
}

// Logic phase for one word of colour c at row r = y + L z, word k (see the
// layout notes in isg_common.cuh), in two halves: word_load issues the loads of
// the word, its forward couplings and the other colour's neighbour words (and
// of the backward couplings there); word_flip counts the unsatisfied bonds, forms
// the flip mask from the draws' levels, writes the word and adds its dE to dEsum.
template <typename Word>
struct WordIn {
    size_t o;
    int p;
    Word s, na, jxc, jyc, jzc, syp, jym, sym, szp, jzm, szm, jxn, jxb, sb;
};

// With CG the other colour's spins are read from L2, past an L1 that may hold
// what they were two passes ago (launches whose passes follow one another
// without a kernel boundary).
template <bool CG, typename Word>
__device__ __forceinline__ Word ld_spin(const Word* p) {
    if constexpr (CG) return __ldcg(p);
    else return *p;
}

template <typename Word, bool CG = false>
__device__ __forceinline__ void word_load(const FlipArgs& a, int c, int r, int y, int z, int k, WordIn<Word>& q) {
    const int L = a.L, W = a.W;
    const size_t pb = (size_t)a.plane_bytes;
    const Word* Sc = (const Word*)(a.planes + (size_t)(4 * c) * pb);
    const Word* Jxc = (const Word*)(a.planes + (size_t)(4 * c + 1) * pb);
    const Word* Jyc = (const Word*)(a.planes + (size_t)(4 * c + 2) * pb);
    const Word* Jzc = (const Word*)(a.planes + (size_t)(4 * c + 3) * pb);
    const int n = c ^ 1;
    const Word* Sn = (const Word*)(a.planes + (size_t)(4 * n) * pb);
    const Word* Jxn = (const Word*)(a.planes + (size_t)(4 * n + 1) * pb);
    const Word* Jyn = (const Word*)(a.planes + (size_t)(4 * n + 2) * pb);
    const Word* Jzn = (const Word*)(a.planes + (size_t)(4 * n + 3) * pb);

    q.p = (c + y + z) & 1;
    const int rowW = r * W;
    const int dym = (y == 0 ? L - 1 : -1) * W, dyp = (y == L - 1 ? 1 - L : 1) * W;
    const int LW = L * W;
    const int dzm = (z == 0 ? (L - 1) * LW : -LW), dzp = (z == L - 1 ? -(L - 1) * LW : LW);
    q.o = (size_t)(rowW + k);
    // the x neighbour word across the word boundary: k - 1 for p = 0, k + 1 for p = 1
    const size_t onb = (size_t)(rowW + (q.p == 0 ? (k == 0 ? W - 1 : k - 1) : (k == W - 1 ? 0 : k + 1)));
    const size_t o = q.o;
    q.s = Sc[o];
    q.na = ld_spin<CG>(Sn + o);
    q.jxc = Jxc[o];
    q.jyc = Jyc[o];
    q.jzc = Jzc[o];
    q.syp = ld_spin<CG>(Sn + o + dyp);
    q.jym = Jyn[o + dym];
    q.sym = ld_spin<CG>(Sn + o + dym);
    q.szp = ld_spin<CG>(Sn + o + dzp);
    q.jzm = Jzn[o + dzm];
    q.szm = ld_spin<CG>(Sn + o + dzm);
    q.jxn = Jxn[o];
    q.jxb = q.p == 0 ? Jxn[onb] : Word(0);
    q.sb = ld_spin<CG>(Sn + onb);
}

template <typename Word>
__device__ __forceinline__ void word_flip(const FlipArgs& a, int c, const WordIn<Word>& q, int k, Word lo, Word hi,
                                          int& dEsum, int* usum = nullptr) {
    constexpr int w = 8 * sizeof(Word);
    const int W = a.W, nt = a.nt;
    Word* Sc = (Word*)(a.planes + (size_t)(4 * c) * (size_t)a.plane_bytes);
    const Word s = q.s, na = q.na;
    const Word e_yp = q.jyc ^ s ^ q.syp;
    const Word e_ym = q.jym ^ s ^ q.sym;
    const Word e_zp = q.jzc ^ s ^ q.szp;
    const Word e_zm = q.jzm ^ s ^ q.szm;
    Word e_xp, e_xm;
    if (q.p == 0) {
        e_xp = q.jxc ^ s ^ na;
        e_xm = row_down<Word>(q.jxn ^ na, q.jxb ^ q.sb, k, nt) ^ s;
    } else {
        e_xp = q.jxc ^ s ^ row_up<Word>(na, q.sb, k, W, nt);
        e_xm = q.jxn ^ s ^ na;
    }
    Word u0, u1, u2;
    Logic<Word>::count6(e_xp, e_xm, e_yp, e_ym, e_zp, e_zm, u0, u1, u2);
    Word f = Logic<Word>::flip(u0, u1, u2, lo | hi, hi, lo & hi);
    const Word valid = (k == W - 1 && nt < w) ? (Word)((Word(1) << nt) - 1) : ~Word(0);
    f &= valid;
    Sc[q.o] = s ^ f;
    dEsum += Logic<Word>::dE(f, u0, u1, u2);
    // the pass's unsatisfied bonds before any flip: every bond has one site of
    // each colour, so their sum over one colour's sites is U of Eq. 1 (E = 2U - 3N)
    if (usum)
        *usum += Logic<Word>::popc(u0 & valid) + 2 * Logic<Word>::popc(u1 & valid) +
                 4 * Logic<Word>::popc(u2 & valid);
}

// Generator state of the stream a warp is working on.
struct StreamRegs {
    int pos;       // MT19937: position (mod 624) of the next draw in the stored ring
    int iA;        // MT19937: window index of x_k for the next draw k
    uint32_t xA;   // MINSTD: state of draw n + lane + 1; Parisi-Rapuano: ira[i-64+lane]
    uint32_t xB;   // MINSTD: state of draw n + lane + 33; Parisi-Rapuano: ira[i-32+lane]
};

// The stored MT19937 state is a 624-word ring with the position of the next
// draw; it is unrolled into the front of the window on load and rolled back on
// store, so the stored format does not depend on the window.
template <int KIND>
__device__ __forceinline__ void load_stream(const FlipArgs& a, int64_t t, uint32_t* B, StreamRegs& st,
                                            const StreamConst& k, int lane) {
    if (KIND == ISG_RNG_MT19937) {
        const int p = (int)a.rng_pos[t];
        for (int j = lane; j < kMtN; j += 32) {
            const int s = p + j >= kMtN ? p + j - kMtN : p + j;
            B[j] = a.rng[t * kMtN + s];
        }
        st.pos = p;
        st.iA = 0;
        __syncwarp();
    } else if (KIND == ISG_RNG_PARISI_RAPUANO) {
        pr_load(a.rng + t * kPrN, st.xA, st.xB, lane);
    } else {
        st.xA = minstd_mulmod(a.rng[t], a.mt.pow[lane + 1]);
        st.xB = minstd_mulmod(st.xA, k.a32);
    }
}

template <int KIND>
__device__ __forceinline__ void store_stream(const FlipArgs& a, int64_t t, const uint32_t* B,
                                             const StreamRegs& st, int lane) {
    if (KIND == ISG_RNG_MT19937) {
        __syncwarp();
        for (int j = lane; j < kMtN; j += 32) {
            const int s = st.pos + j >= kMtN ? st.pos + j - kMtN : st.pos + j;
            a.rng[t * kMtN + s] = B[st.iA + j];
        }
        if (lane == 0) a.rng_pos[t] = (uint32_t)st.pos;
        __syncwarp();
    } else if (KIND == ISG_RNG_PARISI_RAPUANO) {
        pr_store(a.rng + t * kPrN, st.xA, st.xB, lane);
    } else {
        const uint32_t x0 = __shfl_sync(kFull, st.xA, 0);
        if (lane == 0) a.rng[t] = minstd_mulmod(x0, a.mt.inv);  // state of the last draw used
    }
}

// Level of a draw against the nested thresholds, as the two ballot bits.
__device__ __forceinline__ bool level_lo(uint32_t d, const Cmp& a) {
    return (d < a.c1) ^ (d < a.c2) ^ (d < a.c3);
}

// The two ballots of N consecutive 32-draw blocks.
template <int N>
__device__ __forceinline__ void level_ballots(const uint32_t (&d)[N], const Cmp& a, uint32_t (&lo)[N],
                                              uint32_t (&hi)[N]) {
#pragma unroll
    for (int j = 0; j < N; ++j) {
        lo[j] = __ballot_sync(kFull, level_lo(d[j], a));
        hi[j] = __ballot_sync(kFull, d[j] < a.c2);
    }
}

// 16-byte shared-memory store by lane 0 alone, as one predicated instruction
// (no divergent branch around it); `addr` is a shared-window address.
__device__ __forceinline__ void st_shared_lane0(uint32_t addr, uint32_t x, uint32_t y, uint32_t z, uint32_t w,
                                                int lane) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.eq.s32 p, %5, 0;\n\t@p st.shared.v4.u32 [%0], {%1, %2, %3, %4};\n\t}"
        :
        : "r"(addr), "r"(x), "r"(y), "r"(z), "r"(w), "r"(lane)
        : "memory");
}

// The ballots of a quad of blocks (MINSTD and Parisi-Rapuano).  A draw below cmp2
// has probability exp(-8 beta) (1.4e-4 at T = 0.9), so the warp first asks whether
// any of its 128 draws is below cmp2.  If none is, none is below cmp3 either,
// every level is 0 or 1, one comparison per draw gives it exactly and the hi
// ballots are all zero.  Lane 0 stores the four lo ballots at lo and, only when
// the hi ballots are taken, the four hi ballots at hi; returns whether it did.
// The hi stream is otherwise left as it is (kept all zero by the caller).  Stored
// under a branch: for these generators faster than as a predicated instruction.
__device__ __forceinline__ bool quad_ballots(const uint32_t (&d)[4], const Cmp& a, uint32_t* lo, uint32_t* hi,
                                             int lane) {
    const uint32_t dmin = min(min(d[0], d[1]), min(d[2], d[3]));
    if (__any_sync(kFull, dmin < a.c2)) {
        uint32_t l[4], h[4];
        level_ballots<4>(d, a, l, h);
        if (lane == 0) {
            *(uint4*)lo = make_uint4(l[0], l[1], l[2], l[3]);
            *(uint4*)hi = make_uint4(h[0], h[1], h[2], h[3]);
        }
        return true;
    }
    uint32_t l[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) l[j] = __ballot_sync(kFull, d[j] < a.c1);
    if (lane == 0) *(uint4*)lo = make_uint4(l[0], l[1], l[2], l[3]);
    return false;
}

// Zeroes the hi bit stream of the condition buffer (n words).
__device__ __forceinline__ void clear_hi(uint32_t* hi, int n, int lane) {
    for (int j = lane; j < n; j += 32) hi[j] = 0u;
}

// Four consecutive draws a lane against 32 consecutive ones a block and lane (four
// loads and a store against sixteen accesses, one comparison whose result needs
// no vote, no last tempering step): 31.9 -> 29.9 warp instructions per 32
// attempts at L = 1024, 1.054 -> 1.011 ps per attempt (L = 512 1.274 -> 1.217, the
// 512 x 2 batch's pass launches 1.210 -> 1.137; 0.978, 1.156 and 1.090 now).  The shared-memory pipe is then
// 75 % busy, the logic pipe 66 %, issue 74 %.  Two quads a turn of the loop, or
// the multipliers held in registers, changed nothing or lost 1 %.
//
// The MT19937 draws of a row group as level bytes (take_levels) in `lv`: the
// group's first draw is draw off0 (< 16) of the array, of whose draws the first
// `have` (a multiple of 16) were made with the last group's; makes whole quads
// until need = off0 + the group's draws are there.
template <int SLACK, bool REDUX>
__device__ __forceinline__ void mt_group_levels(uint32_t* B, int& iA, uint32_t* lv, int& have, int need, const Cmp& cm,
                                                const Cmp4& c4, const MtMul& k, int lane) {
    while (have < need) {
        mt_make_room<SLACK>(B, iA, 128, lane);
        const int fit = (mt_window(SLACK) - kMtN - iA) >> 7, want = (need - have + 127) >> 7;
        unsigned char* at = (unsigned char*)lv + have / 4 + lane;
        for (int q = fit < want ? fit : want; q > 0; --q) {
            uint32_t v[4];
            mt_quad4(B, iA, v, k, lane);
            *at = (unsigned char)mt_level_finish<REDUX>(mt_level_begin(v, c4, k), cm, c4);
            at += 32;
            have += 128;
        }
    }
}

// One pass of colour c over rows [r_begin, r_end) of a stream; the generator
// state, positioned at the first of these rows, is in B / st.  SLACK is the free
// space of the MT19937 window (see mt_window).  WPT is the number of words of a
// row group each lane updates: a group is WPT * 32 / W rows, and cond holds its
// levels: two bit streams of WPT * kCondWords words each, or (MT19937) level
// bytes in the same space, 16 draws a word.
template <typename Word, int KIND, int SLACK, int WPT = 1, bool REDUX = false>
__device__ __forceinline__ void stream_pass(const FlipArgs& a, int c, int64_t r_begin, int64_t r_end, uint32_t* B,
                                            uint32_t* cond, StreamRegs& st, const StreamConst& k, int lane,
                                            int& dEsum, int* usum = nullptr) {
    constexpr int w = 8 * sizeof(Word);
    constexpr bool kMT = KIND == ISG_RNG_MT19937;
    constexpr int kCond = WPT * kCondWords;
    // A group has at most 32 WPT words of 64 draws; up to 15 draws precede its first
    // one in the level bytes, and the quad that completes it makes up to 127 more.
    // (A window of take_levels starts at one of the group's draws and reads four
    // words on.)
    static_assert((2048 * WPT + 15 + 127) / 16 <= 2 * kCond && (2048 * WPT + 14) / 16 + 4 < 2 * kCond,
                  "the level bytes of a row group fit");
    const int W = a.W, half = a.half, L = a.L;
    const Cmp cm = cmp_of(a);
    const Cmp4 c4 = cmp4_of(cm);
    const int G = WPT * 32 / W;
    const int lj = lane / W, lk = lane - lj * W;
    const int loff = lj * half + lk * w;
    int r = (int)r_begin + lj;
    int y = r % L, z = r / L;
    bool hiset = false;  // the hi stream holds a nonzero word
    // MT19937: whole quads are made, whatever the groups' draws: draws past a
    // group's end are kept as levels for the next one, of those past the pass's end
    // the window still holds the words
    int off0 = 0, have = 0;
    if (kMT) {
        const int total = (int)(r_end - r_begin) * half;
        if (st.iA & 3) mt_make_room<SLACK>(B, st.iA, SLACK + 1, lane);  // to a multiple of 4
        st.pos = (st.pos + total) % kMtN;
    } else {
        clear_hi(cond + kCond, kCond, lane);
        __syncwarp();
    }
    auto update = [&](int rq, int yq, int zq, int kq, int off) {
        WordIn<Word> q;
        word_load<Word>(a, c, rq, yq, zq, kq, q);
        Word lo, hi;
        if constexpr (kMT) {
            take_levels<Word>(cond, off0 + off, lo, hi);
        } else {
            lo = take_bits<Word>(cond, off);
            hi = take_bits<Word>(cond + kCond, off);
        }
        word_flip<Word>(a, c, q, kq, lo, hi, dEsum, usum);
    };
    for (int64_t g0 = r_begin; g0 < r_end; g0 += G) {
        const int nrows = (int)((r_end - g0) < G ? (r_end - g0) : G);
        const int D = nrows * half;
        if constexpr (kMT) {
            mt_group_levels<SLACK, REDUX>(B, st.iA, cond, have, off0 + D, cm, c4, k.mul, lane);
        } else {
            // draws four 32-draw blocks per step, then the remaining blocks one by
            // one.  The hi stream is kept all zero between groups and a quad whose
            // hi ballots were skipped stores nothing there.
            // Not unrolled: MINSTD L = 1024 0.544 -> 0.523 ps, L = 512 0.709 -> 0.694
            // (Parisi-Rapuano the same).
            const int nquads = D >> 7;
#pragma unroll 1
            for (int q = 0; q < nquads; ++q) {
                uint32_t d[4];
                if (KIND == ISG_RNG_PARISI_RAPUANO) {
#pragma unroll
                    for (int j = 0; j < 4; ++j) d[j] = pr_warp_step(st.xA, st.xB, lane, 32);
                } else {
                    d[0] = st.xA;
                    d[1] = st.xB;
                    d[2] = minstd_mulmod(st.xA, k.a64);
                    d[3] = minstd_mulmod(st.xB, k.a64);
                    st.xA = minstd_mulmod(d[2], k.a64);
                    st.xB = minstd_mulmod(d[3], k.a64);
                }
                if (quad_ballots(d, cm, cond + 4 * q, cond + kCond + 4 * q, lane)) hiset = true;
            }
            int b = 4 * nquads;
            for (int rem = D - 32 * b; rem > 0; rem -= 32, ++b) {
                const int nvalid = rem < 32 ? rem : 32;
                uint32_t d;
                if (KIND == ISG_RNG_PARISI_RAPUANO) {
                    d = pr_warp_step(st.xA, st.xB, lane, nvalid);
                } else {
                    d = st.xA;
                    const int src = lane + nvalid;
                    const uint32_t pa = __shfl_sync(kFull, st.xA, src & 31);
                    const uint32_t pb = __shfl_sync(kFull, st.xB, src & 31);
                    st.xA = src < 32 ? pa : pb;
                    st.xB = minstd_mulmod(st.xA, k.a32);
                }
                const uint32_t lo = __ballot_sync(kFull, level_lo(d, cm));
                const uint32_t hi = __ballot_sync(kFull, d < cm.c2);
                hiset |= hi != 0u;
                if (lane == 0) {
                    cond[b] = lo;
                    cond[kCond + b] = hi;
                }
            }
        }
        __syncwarp();
        if constexpr (WPT == 1) {
            if (lane < nrows * W) update(r, y, z, lk, loff);
        } else {
#pragma unroll
            for (int q = 0; q < WPT; ++q) {
                const int wi = lane + 32 * q;  // word of the group: row wi / W, word wi % W
                if (wi < nrows * W) {
                    const int jq = wi / W, kq = wi - jq * W;
                    const int rq = (int)g0 + jq;
                    update(rq, rq % L, rq / L, kq, jq * half + kq * w);
                }
            }
        }
        __syncwarp();
        if constexpr (kMT) {
            // the levels past the group's end to the front (at most 9 words)
            const int end = off0 + D, first = end >> 4, left = (have >> 4) - first;
            off0 = end & 15;
            have = 16 * left;
            if (left > 0) {
                const uint32_t v = cond[first + (lane < left ? lane : 0)];
                __syncwarp();
                if (lane < left) cond[lane] = v;
                __syncwarp();
            }
        } else if (hiset) {
            clear_hi(cond + kCond, kCond, lane);
            hiset = false;
            __syncwarp();
        }
        r += G;
        y += G;
        while (y >= L) {
            y -= L;
            ++z;
        }
    }
    // Back to the first draw not used.  It is one of the last quad's 128 (nothing is
    // made past the quad that ends a pass), and a window that moved did so before
    // that quad: iA stays at or behind the window's front.  (Moves that kept 128 words
    // before the live ones, for streams of other than whole quads, needed them for
    // nothing: L = 1024 0.998 -> 0.978 ps per attempt without them, L = 512 1.218 ->
    // 1.156, the 512 x 2 batch 122.7 -> 118.0 ms.)
    if (kMT) st.iA -= have - off0;
}

}  // namespace isg
