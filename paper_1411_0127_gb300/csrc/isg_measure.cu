// isg_measure.cu -- popcount kernels for the energy (Eq. 1), the replica
// overlap and the Zobrist hash, and the kernels that convert the coupling planes
// to and from int8 +-1 arrays in site order i = x + L*y + L*L*z (the spins'
// conversions are in isg_spinio.cu).
//
// Energy: every coupling is the forward (+x, +y or +z) coupling of exactly one
// site, so U = number of unsatisfied bonds = sum over both colours and all words
// of popc(e_+x) + popc(e_+y) + popc(e_+z), with e = J ^ s ^ s' (Sec. 4 bit map),
// and E = 2U - 3N.
#include <algorithm>

#include "isg_common.cuh"

namespace isg {

struct MeasGeom {
    const unsigned char* planes;
    int64_t plane_bytes;
    int L, half, W, nt;
    int64_t rows;
};

static MeasGeom mgeom(const isg_sim* h) {
    MeasGeom g;
    g.planes = h->planes;
    g.plane_bytes = h->plane_bytes;
    g.L = h->L;
    g.half = h->half;
    g.W = h->W;
    g.nt = h->nt;
    g.rows = h->rows;
    return g;
}

template <typename Word>
__device__ __forceinline__ const Word* plane(const MeasGeom& g, int c, int q) {
    return (const Word*)(g.planes + (size_t)(4 * c + q) * g.plane_bytes);
}

template <typename Word>
__device__ __forceinline__ Word valid_mask(const MeasGeom& g, int k) {
    constexpr int w = 8 * sizeof(Word);
    return (k == g.W - 1 && g.nt < w) ? (Word)((Word(1) << g.nt) - 1) : ~Word(0);
}

__device__ __forceinline__ int popcw(uint32_t v) { return __popc(v); }
__device__ __forceinline__ int popcw(uint64_t v) { return __popcll(v); }

// Where a measuring kernel's sum goes: added to the device word `out`, or, with
// out == NULL, gathered in the handle's words acc and count (both zero between
// calls) and written to pinned host memory by the last block to finish, together
// with the handle's error word: no clearing before the kernel and no copy after
// it, so a call is one launch and one wait (with the clearing and the copy,
// isg_overlap took 50 us at L = 512, now 28.5).
struct Finish {
    unsigned long long* out;
    unsigned long long *acc, *count;
    const long long* err;
    unsigned long long* host;  // [0] the sum, [1] the error word
};

static Finish finish_to(long long* out) { return Finish{(unsigned long long*)out, nullptr, nullptr, nullptr, nullptr}; }
static Finish finish_on_host(const isg_sim* h, unsigned long long* host) {
    unsigned long long* w = (unsigned long long*)h->scal;
    return Finish{nullptr, w + 6, w + 7, h->scal + 5, host};
}

// Sum (XOR: exclusive or) of v over the block in thread 0.
template <bool XOR>
__device__ __forceinline__ unsigned long long block_sum(unsigned long long v) {
    __shared__ unsigned long long part[32];
    for (int sh = 16; sh; sh >>= 1) {
        const unsigned long long o = __shfl_xor_sync(kFull, v, sh);
        v = XOR ? v ^ o : v + o;
    }
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x == 0)
        for (unsigned i = 1; i < (blockDim.x + 31) / 32; ++i) v = XOR ? v ^ part[i] : v + part[i];
    return v;
}

template <bool XOR>
__device__ __forceinline__ void finish(const Finish& f, unsigned long long v) {
    v = block_sum<XOR>(v);
    if (threadIdx.x != 0) return;
    unsigned long long* to = f.out ? f.out : f.acc;
    if (v) {
        if (XOR) atomicXor(to, v);
        else atomicAdd(to, v);
    }
    if (f.out) return;
    __threadfence();
    if (atomicAdd(f.count, 1ull) == gridDim.x - 1) {
        __threadfence();
        f.host[0] = atomicExch(f.acc, 0ull);
        f.host[1] = (unsigned long long)*f.err;
        *f.count = 0ull;
    }
}

static unsigned grid_for(int64_t n, int threads) {
    int64_t b = (n + threads - 1) / threads;
    if (b > 152 * 32) b = 152 * 32;
    if (b < 1) b = 1;
    return (unsigned)b;
}

// ---------------------------------------------------------------- energy ---
// Thread t of a block owns word k = t % W of rows r = t / W + rows_per_block * j
// (blocks striding over rows) and counts the forward bonds of that word in BOTH
// colours, so every plane is read from memory once: the neighbour words of one
// colour's word (rows y+1 and z+1 of the other colour, and the next word of the
// row for the site whose +x neighbour is shifted) are words another thread of
// the same pass reads as its own, found in L1 or L2.
template <typename Word>
struct UnsatPair {
    Word s0, s1, jx0, jy0, jz0, jx1, jy1, jz1, n1y, n1z, n0y, n0z, nb;
    int p0;
};

template <typename Word>
__device__ __forceinline__ void unsat_pair_load(const MeasGeom& g, int r, int y, int z, int k, UnsatPair<Word>& u) {
    const int L = g.L, W = g.W;
    const size_t o = (size_t)r * W + k;
    const int ryp = y == L - 1 ? r - (L - 1) : r + 1;
    const int rzp = z == L - 1 ? r - (L - 1) * L : r + L;
    const Word* S0 = plane<Word>(g, 0, 0);
    const Word* S1 = plane<Word>(g, 1, 0);
    u.p0 = (y + z) & 1;  // colour 0's row parity; colour 1's is the other
    u.s0 = S0[o];
    u.s1 = S1[o];
    u.jx0 = plane<Word>(g, 0, 1)[o];
    u.jy0 = plane<Word>(g, 0, 2)[o];
    u.jz0 = plane<Word>(g, 0, 3)[o];
    u.jx1 = plane<Word>(g, 1, 1)[o];
    u.jy1 = plane<Word>(g, 1, 2)[o];
    u.jz1 = plane<Word>(g, 1, 3)[o];
    u.n1y = S1[(size_t)ryp * W + k];
    u.n1z = S1[(size_t)rzp * W + k];
    u.n0y = S0[(size_t)ryp * W + k];
    u.n0z = S0[(size_t)rzp * W + k];
    // the colour whose row parity is 1 has its +x neighbours shifted by one site
    const size_t onb = (size_t)r * W + (k == W - 1 ? 0 : k + 1);
    u.nb = (u.p0 == 1 ? S1 : S0)[onb];
}

template <typename Word>
__device__ __forceinline__ int unsat_pair_count(const MeasGeom& g, int k, const UnsatPair<Word>& u) {
    const Word m = valid_mask<Word>(g, k);
    const Word nx0 = u.p0 == 1 ? row_up<Word>(u.s1, u.nb, k, g.W, g.nt) : u.s1;
    const Word nx1 = u.p0 == 1 ? u.s0 : row_up<Word>(u.s0, u.nb, k, g.W, g.nt);
    return popcw((u.jx0 ^ u.s0 ^ nx0) & m) + popcw((u.jy0 ^ u.s0 ^ u.n1y) & m) +
           popcw((u.jz0 ^ u.s0 ^ u.n1z) & m) + popcw((u.jx1 ^ u.s1 ^ nx1) & m) +
           popcw((u.jy1 ^ u.s1 ^ u.n0y) & m) + popcw((u.jz1 ^ u.s1 ^ u.n0z) & m);
}

// Rows advance by `step` per iteration: (y, z) follow with the precomputed
// step % L and step / L and one carry.
__device__ __forceinline__ void row_advance(int& r, int& y, int& z, int step, int sy, int sz, int L) {
    r += step;
    y += sy;
    z += sz;
    if (y >= L) {
        y -= L;
        ++z;
    }
}

// Rows first, first + step, ... below `end` for this thread's word slot.
template <typename Word>
__device__ __forceinline__ unsigned unsat_rows(const MeasGeom& g, int first, int step, int rows) {
    const int L = g.L, W = g.W;
    const int rpb = blockDim.x / W;  // rows per block and iteration
    const int t = threadIdx.x;
    const int rl = t / W, k = t - rl * W;
    unsigned acc = 0;
    if (rl < rpb) {
        const int sy = step % L, sz = step / L;
        int r = first + rl;
        int y = r % L, z = r / L;
        // two rows in flight: all their loads are issued before either is counted
        while (r < rows) {
            int r2 = r, y2 = y, z2 = z;
            row_advance(r2, y2, z2, step, sy, sz, L);
            UnsatPair<Word> a, b;
            unsat_pair_load<Word>(g, r, y, z, k, a);
            const bool two = r2 < rows;
            if (two) unsat_pair_load<Word>(g, r2, y2, z2, k, b);
            acc += unsat_pair_count<Word>(g, k, a);
            if (two) acc += unsat_pair_count<Word>(g, k, b);
            r = r2;
            y = y2;
            z = z2;
            row_advance(r, y, z, step, sy, sz, L);
        }
    }
    return acc;
}

template <typename Word>
__global__ void unsat_kernel(MeasGeom g, Finish f) {
    const int rpb = blockDim.x / g.W;
    finish<false>(f, unsat_rows<Word>(g, blockIdx.x * rpb, gridDim.x * rpb, (int)g.rows));
}

static cudaError_t launch_unsat(const isg_sim* h, const Finish& f, cudaStream_t s) {
    const MeasGeom g = mgeom(h);
    const int threads = 256;
    const int64_t rpb = threads / h->W;
    int64_t blocks = (h->rows + rpb - 1) / rpb;
    const int64_t cap = (int64_t)sm_count() * 8;
    if (blocks > cap) blocks = cap;
    if (h->wbits == 64) unsat_kernel<uint64_t><<<(unsigned)blocks, threads, 0, s>>>(g, f);
    else unsat_kernel<uint32_t><<<(unsigned)blocks, threads, 0, s>>>(g, f);
    return cudaGetLastError();
}

cudaError_t launch_energy(const isg_sim* h, long long* out, cudaStream_t s) {
    return launch_unsat(h, finish_to(out), s);
}
cudaError_t launch_energy_host(const isg_sim* h, unsigned long long* host, cudaStream_t s) {
    return launch_unsat(h, finish_on_host(h, host), s);
}

// --------------------------------------------------------------- overlap ---
// Number of sites where the two replicas differ (tail bits are zero in both).
__global__ void differ_kernel(const ulonglong2* a0, const ulonglong2* a1, const ulonglong2* b0, const ulonglong2* b1,
                              int64_t n, Finish f) {
    unsigned acc = 0;
    for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < n; q += (int64_t)gridDim.x * blockDim.x) {
        const ulonglong2 u = a0[q], v = b0[q], x = a1[q], y = b1[q];
        acc += __popcll(u.x ^ v.x) + __popcll(u.y ^ v.y) + __popcll(x.x ^ y.x) + __popcll(x.y ^ y.y);
    }
    finish<false>(f, acc);
}

cudaError_t launch_overlap_host(const isg_sim* a, const isg_sim* b, unsigned long long* host, cudaStream_t s) {
    const int64_t n = a->plane_bytes / 16;  // planes are multiples of 256 bytes
    int64_t blocks = (n + 255) / 256;
    blocks = std::max<int64_t>(1, std::min<int64_t>(blocks, (int64_t)sm_count() * 8));
    differ_kernel<<<(unsigned)blocks, 256, 0, s>>>((const ulonglong2*)a->plane(0, 0), (const ulonglong2*)a->plane(1, 0),
                                                   (const ulonglong2*)b->plane(0, 0), (const ulonglong2*)b->plane(1, 0),
                                                   n, finish_on_host(a, host));
    return cudaGetLastError();
}

// ------------------------------------------------------------------ hash ---
// SplitMix64 of the 32 sites i0, i0 + 2, ..., i0 + 62, exclusive-or of those whose
// bit in v is set, without the finaliser's last step z ^= z >> 31: that step is
// linear over exclusive or, so it is applied once, to the total (hash_finish).
// All sites are computed and masked: following the set bits alone (half of them)
// costs a find-first and a 64-bit clear each, and lanes with fewer bits wait
// (isg_hash at L = 512: 175 us that way, 134 now; integer issue bounds both).
// From the highest site down, so that the mask is v's sign.
__device__ __forceinline__ void hash32(uint64_t i0, uint32_t v, uint32_t& lo, uint32_t& hi) {
    constexpr uint64_t kStep = 0x9E3779B97F4A7C15ull;
    uint64_t st = kSaltHash + (i0 + 63ull) * kStep;
#pragma unroll 8
    for (int b = 0; b < 32; ++b) {
        uint64_t z = st;
        z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
        z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
        const uint32_t m = (uint32_t)((int32_t)v >> 31);
        lo ^= (uint32_t)z & m;
        hi ^= (uint32_t)(z >> 32) & m;
        v += v;
        st -= 2 * kStep;
    }
}

uint64_t hash_finish(uint64_t x) { return x ^ (x >> 31); }

// Units of 32 bits: unit q of colour c is bits 32 u .. 32 u + 31 of row r.
template <typename Word>
__device__ __forceinline__ unsigned long long hash_units(const MeasGeom& g, unsigned first, unsigned step, unsigned end) {
    constexpr unsigned kPer = sizeof(Word) / 4;
    const unsigned per = (unsigned)g.W * kPer, all = (unsigned)g.rows * per, L = (unsigned)g.L;
    uint32_t lo = 0, hi = 0;
    for (unsigned q = first; q < end; q += step) {
        const unsigned c = q >= all, o = q - c * all, r = o / per, u = o - r * per;
        const unsigned z = r / L, y = r - z * L, p = (c + y + z) & 1u;
        // bits past L / 2 are zero
        const uint32_t v = ((const uint32_t*)plane<Word>(g, (int)c, 0))[o];
        if (v) hash32((uint64_t)r * L + 64ull * u + p, v, lo, hi);
    }
    return ((unsigned long long)hi << 32) | lo;
}

template <typename Word>
__global__ void hash_kernel(MeasGeom g, Finish f) {
    const unsigned n = 2u * (unsigned)g.rows * (unsigned)g.W * (sizeof(Word) / 4);
    finish<true>(f, hash_units<Word>(g, blockIdx.x * blockDim.x + threadIdx.x, gridDim.x * blockDim.x, n));
}

cudaError_t launch_hash_host(const isg_sim* h, unsigned long long* host, cudaStream_t s) {
    const MeasGeom g = mgeom(h);
    const int64_t n = 2 * h->rows * h->W * (h->wbits / 32);
    int64_t blocks = std::max<int64_t>(1, std::min<int64_t>((n + 255) / 256, (int64_t)sm_count() * 8));
    if (h->wbits == 64) hash_kernel<uint64_t><<<(unsigned)blocks, 256, 0, s>>>(g, finish_on_host(h, host));
    else hash_kernel<uint32_t><<<(unsigned)blocks, 256, 0, s>>>(g, finish_on_host(h, host));
    return cudaGetLastError();
}

// ----------------------------------------------------- a batch's replicas ---
// All replicas of a batch in one launch: block b measures chunk b = (replica,
// first row, rows) and adds to its replica's words.  Replicas are in 64-bit
// words; 2 s and 2 s + 1 belong to sample s.  (One call, one copy and one wait a
// replica and quantity took 25.5 ms for the energies and overlaps and 34 ms for
// the tracked energies and hashes of the 512 x 2 batch: 0.31 and 2.06 ms now,
// most of the latter the hashes' integer work on 1.7e9 sites.)
static __device__ MeasGeom geom_of(const FlipArgs& a) {
    MeasGeom g;
    g.planes = a.planes;
    g.plane_bytes = a.plane_bytes;
    g.L = a.L;
    g.half = a.half;
    g.W = a.W;
    g.nt = a.nt;
    g.rows = a.rows;
    return g;
}

__global__ void batch_energy_kernel(const FlipArgs* reps, const int4* chunks, unsigned long long* U) {
    const int4 ch = chunks[blockIdx.x];
    const MeasGeom g = geom_of(reps[ch.x]);
    const unsigned long long v = block_sum<false>(unsat_rows<uint64_t>(g, ch.y, blockDim.x / g.W, ch.y + ch.z));
    if (threadIdx.x == 0 && v) atomicAdd(U + ch.x, v);
}

__global__ void batch_overlap_kernel(const FlipArgs* reps, const int4* chunks, unsigned long long* differ) {
    const int4 ch = chunks[blockIdx.x];
    if (ch.x & 1) return;
    const MeasGeom a = geom_of(reps[ch.x]), b = geom_of(reps[ch.x + 1]);
    unsigned acc = 0;
    for (int q = ch.y * a.W + threadIdx.x; q < (ch.y + ch.z) * a.W; q += blockDim.x)
        acc += __popcll(plane<uint64_t>(a, 0, 0)[q] ^ plane<uint64_t>(b, 0, 0)[q]) +
               __popcll(plane<uint64_t>(a, 1, 0)[q] ^ plane<uint64_t>(b, 1, 0)[q]);
    const unsigned long long v = block_sum<false>(acc);
    if (threadIdx.x == 0 && v) atomicAdd(differ + ch.x / 2, v);
}

__global__ void batch_hash_kernel(const FlipArgs* reps, const int4* chunks, unsigned long long* H) {
    const int4 ch = chunks[blockIdx.x];
    const MeasGeom g = geom_of(reps[ch.x]);
    const unsigned per = 2u * g.W, all = (unsigned)g.rows * per, q0 = ch.y * per, q1 = (ch.y + ch.z) * per;
    const unsigned long long v = block_sum<true>(hash_units<uint64_t>(g, q0 + threadIdx.x, blockDim.x, q1) ^
                                                 hash_units<uint64_t>(g, all + q0 + threadIdx.x, blockDim.x, all + q1));
    if (threadIdx.x == 0 && v) atomicXor(H + ch.x, v);
}

// dE and the error word of every replica (scal[0] and scal[5] of its handle)
__global__ void batch_words_kernel(const FlipArgs* reps, int n, unsigned long long* dE, unsigned long long* err) {
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= n) return;
    const unsigned long long* w = (const unsigned long long*)reps[r].dE;
    dE[r] = w[0];
    err[r] = w[5];
}

cudaError_t launch_batch_measures(const BatchMeasure& m, cudaStream_t s) {
    if (m.U) batch_energy_kernel<<<m.nchunks, 256, 0, s>>>(m.reps, m.chunks, m.U);
    if (m.differ) batch_overlap_kernel<<<m.nchunks, 256, 0, s>>>(m.reps, m.chunks, m.differ);
    if (m.H) batch_hash_kernel<<<m.nchunks, 256, 0, s>>>(m.reps, m.chunks, m.H);
    if (m.dE) batch_words_kernel<<<(m.nreps + 255) / 256, 256, 0, s>>>(m.reps, m.nreps, m.dE, m.err);
    return cudaGetLastError();
}

// ------------------------------------------------------ unpack / pack ---
// q = 0: spins (bit 1 -> +1); q = 1..3: couplings (bit 1 -> -1).
template <typename Word>
__global__ void unpack_kernel(MeasGeom g, int q, int8_t* out) {
    constexpr int w = 8 * sizeof(Word);
    const int64_t L = g.L, N = L * L * L;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < N; i += (int64_t)gridDim.x * blockDim.x) {
        const int x = (int)(i % L), y = (int)((i / L) % L), z = (int)(i / (L * L));
        const int c = (x + y + z) & 1;
        const int h = x >> 1, k = h / w, b = h % w;
        const Word word = plane<Word>(g, c, q)[((size_t)y + (size_t)L * z) * g.W + k];
        const int bit = (int)((word >> b) & 1);
        out[i] = q == 0 ? (bit ? 1 : -1) : (bit ? -1 : 1);
    }
}

template <typename Word>
__global__ void pack_kernel(MeasGeom g, int q, const int8_t* in) {
    constexpr int w = 8 * sizeof(Word);
    const int64_t nw = 2 * g.rows * g.W;
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < nw; t += (int64_t)gridDim.x * blockDim.x) {
        const int c = (int)(t / (g.rows * g.W));
        const int64_t rem = t - (int64_t)c * g.rows * g.W;
        const int r = (int)(rem / g.W);
        const int k = (int)(rem - (int64_t)r * g.W);
        const int L = g.L;
        const int y = r % L, z = r / L;
        const int p = (c + y + z) & 1;
        Word word = 0;
        for (int b = 0; b < w; ++b) {
            const int h = k * w + b;
            if (h >= g.half) break;
            const int64_t i = (int64_t)(2 * h + p) + (int64_t)L * y + (int64_t)L * L * z;
            const int v = in[i];
            const bool one = (q == 0) ? (v == 1) : (v == -1);
            if (one) word |= (Word)1 << b;
        }
        ((Word*)(g.planes + (size_t)(4 * c + q) * g.plane_bytes))[(size_t)r * g.W + k] = word;
    }
}

cudaError_t launch_unpack_couplings(const isg_sim* h, int8_t* out, cudaStream_t s) {
    const MeasGeom g = mgeom(h);
    const int64_t N = (int64_t)h->L * h->L * h->L;
    for (int d = 0; d < 3; ++d) {
        if (h->wbits == 64) unpack_kernel<uint64_t><<<grid_for(N, 256), 256, 0, s>>>(g, 1 + d, out + d * N);
        else unpack_kernel<uint32_t><<<grid_for(N, 256), 256, 0, s>>>(g, 1 + d, out + d * N);
    }
    return cudaGetLastError();
}

cudaError_t launch_pack_couplings(isg_sim* h, const int8_t* in, cudaStream_t s) {
    const MeasGeom g = mgeom(h);
    const int64_t N = (int64_t)h->L * h->L * h->L;
    const int64_t nw = 2 * h->rows * h->W;
    for (int d = 0; d < 3; ++d) {
        if (h->wbits == 64) pack_kernel<uint64_t><<<grid_for(nw, 256), 256, 0, s>>>(g, 1 + d, in + d * N);
        else pack_kernel<uint32_t><<<grid_for(nw, 256), 256, 0, s>>>(g, 1 + d, in + d * N);
    }
    return cudaGetLastError();
}

__global__ void check_pm1_kernel(const int8_t* in, int64_t n, int* bad) {
    int b = 0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        b |= (in[i] != 1 && in[i] != -1);
    if (__any_sync(kFull, b) && (threadIdx.x & 31) == 0) atomicOr(bad, 1);
}

cudaError_t launch_check_pm1(const int8_t* in, int64_t n, int* bad, cudaStream_t s) {
    check_pm1_kernel<<<grid_for(n, 256), 256, 0, s>>>(in, n, bad);
    return cudaGetLastError();
}

}  // namespace isg
