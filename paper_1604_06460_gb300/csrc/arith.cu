// Emulated multiplication and division (Sec. III-A): instead of simulating
// the Toffoli network of a reversible multiplier or divider, the emulator
// evaluates the classical function on every basis state and moves each
// amplitude to its image.  Three registers a, b, c of N qubits (bit j of a
// value <-> qa[j], qb[j], qc[j]):
//   multiplication  c -> (c + a b) mod 2^N      (the paper's (a, b, 0) -> (a, b, ab)),
//   division        the restoring division: for i = N-1 .. 0,
//                   c_i ^= [b != 0 and a >= b 2^i], then a -= b 2^i if c_i = 1
//                   (the paper's (a, b, 0) -> (a mod b, b, a / b)).
// Both maps are permutations of the basis states; amplitudes are moved bit
// for bit, no arithmetic touches them.
//
// Each map is closed on "planes": the multiplication permutes the 2^N values
// of c for fixed a, b and the other qubits; the division permutes the 2^(2N)
// values of (a, c) for fixed b and the other qubits.  Planes of at most 64 KB
// go through shared-memory tiles of 64 KB (several planes a tile, filled up
// with the lowest other qubits so that memory is touched in long runs): one
// read and one write of every amplitude.  Larger planes are scattered into a
// scratch buffer in batches small enough to stay in L2 and copied back.  In
// both, a thread works on many amplitudes of one tile or chunk, so that the
// index arithmetic with the plane's qubits is done once for them, and values
// fit 32 bits: nine-qubit registers at n = 28 in complex128, multiplication
// 2.46 -> 1.48 ms, division (planes of 4 MB; a gather into a buffer of 1 GB
// and a copy back before) 9.4 -> 3.7 ms; one pass over the state is 1.27 ms.
#include <algorithm>
#include <cstring>

#include "qe_arith.cuh"
#include "qe_internal.h"

namespace qe {

namespace {

constexpr int kArithThreads = 512, kWideThreads = 1024;   // of a tile of 64 KB, of 128 KB

struct RegArg {
    int lo;            // qubit of bit 0
    int contiguous;    // qubits lo .. lo + N - 1 in order
    uint8_t q[16];
};

__device__ __forceinline__ uint32_t reg_get(const RegArg& r, int N, uint64_t x) {
    if (r.contiguous) return (uint32_t)(x >> r.lo) & ((1u << N) - 1u);
    uint32_t v = 0;
    for (int j = 0; j < N; ++j) v |= (uint32_t)((x >> r.q[j]) & 1u) << j;
    return v;
}
__device__ __forceinline__ uint64_t reg_put(const RegArg& r, int N, uint32_t v) {
    if (r.contiguous) return (uint64_t)v << r.lo;
    uint64_t x = 0;
    for (int j = 0; j < N; ++j) x |= (uint64_t)((v >> j) & 1u) << r.q[j];
    return x;
}

enum { kMul = 0, kDiv = 1 };

// The inverse map on register values: the preimage of (a, b, c) in *a, *c.
// Multiplication: c - a b mod 2^N (products wrap mod 2^32 alike).  Division: the
// restoring steps undone in reverse order (i = 0 .. N-1): if c_i, a += b 2^i;
// then c_i ^= [b != 0 and a >= b 2^i] (b 2^i < 2^32).
template <int OP>
__device__ __forceinline__ void preimage(int N, uint32_t& a, uint32_t b, uint32_t& c) {
    const uint32_t mask = (1u << N) - 1u;
    if (OP == kMul) {
        c = (c - a * b) & mask;
        return;
    }
    if (b == 0u) {       // no step adds or flips anything
        return;
    }
    uint32_t bi = b;
    for (int i = 0; i < N; ++i, bi <<= 1) {
        const uint32_t bit = 1u << i;
        if (c & bit) a = (a + bi) & mask;
        if (a >= bi) c ^= bit;
    }
}

// The division itself: the image of (a, b, c) in a, c.
__device__ __forceinline__ void image(int N, uint32_t& a, uint32_t b, uint32_t& c) {
    const uint32_t mask = (1u << N) - 1u;
    if (b == 0u) {       // c_i set subtracts nothing
        return;
    }
    uint32_t bi = b << (N - 1);
    for (int i = N - 1; i >= 0; --i, bi >>= 1) {
        const uint32_t bit = 1u << i;
        if (a >= bi) c ^= bit;
        if (c & bit) a = (a - bi) & mask;
    }
}

template <class S>
struct TileArgs {
    S* x;
    uint64_t ntiles;
    int N, T, L, kh;          // tile of 2^T amplitudes: runs of 2^L, kh bits at or above L
    uint8_t hq[16];
    RegArg a, b;              // by global qubits
    RegArg la, lc;            // by tile-local bits (la: division)
};

// Whole planes in shared memory: one read and one write per amplitude.
template <class S, int OP, int TH>
__global__ void __launch_bounds__(TH) k_arith_plane(const __grid_constant__ TileArgs<S> a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    S* buf = reinterpret_cast<S*>(smem_raw);
    __shared__ uint64_t offA[64], offB[256];
    if (threadIdx.x < 256) {
        uint64_t oa = 0, ob = 0;
        for (int j = 0; j < a.kh; ++j)
            if (j < 6) oa |= ((uint64_t)(threadIdx.x >> j) & 1ull) << a.hq[j];
            else ob |= ((uint64_t)(threadIdx.x >> (j - 6)) & 1ull) << a.hq[j];
        if (threadIdx.x < 64) offA[threadIdx.x] = oa;
        offB[threadIdx.x] = ob;
    }
    __syncthreads();
    const uint32_t E = 1u << a.T, lowmask = (1u << a.L) - 1u;
    const uint32_t cmask = (uint32_t)reg_put(a.lc, a.N, (1u << a.N) - 1u);
    const uint32_t amask = OP == kDiv ? (uint32_t)reg_put(a.la, a.N, (1u << a.N) - 1u) : 0u;
    for (uint64_t t = blockIdx.x; t < a.ntiles; t += gridDim.x) {
        const uint64_t base = insert_zero_bits(t << a.L, a.hq, a.kh);
        auto at = [&](uint32_t i) { return base + (i & lowmask) + offA[(i >> a.L) & 63u] + offB[i >> a.L >> 6]; };
#pragma unroll 8
        for (uint32_t i = threadIdx.x; i < E; i += TH) buf[i] = a.x[at(i)];
        __syncthreads();
#pragma unroll 4
        for (uint32_t i = threadIdx.x; i < E; i += TH) {
            const uint64_t x = at(i);
            const uint32_t bv = reg_get(a.b, a.N, x);
            uint32_t av = OP == kDiv ? reg_get(a.la, a.N, i) : reg_get(a.a, a.N, x);
            uint32_t cv = reg_get(a.lc, a.N, i);
            preimage<OP>(a.N, av, bv, cv);
            uint32_t src = (i & ~(cmask | amask)) | (uint32_t)reg_put(a.lc, a.N, cv);
            if (OP == kDiv) src |= (uint32_t)reg_put(a.la, a.N, av);
            a.x[x] = buf[src];
        }
        __syncthreads();
    }
}

// Larger planes: of divisions only (registers have at most 11 qubits, and 2^11
// values of c are 32 KB).  A block is 2^w planes that differ in the lowest w <= 3 qubits
// (those below every plane qubit), its value e = (plane value y) 2^w + (low
// bits l), so that a warp touches whole lines of the state wherever the
// registers lie.
template <class S>
struct ArithArgs {
    S* x;
    S* scratch;                 // blocks [blk0, blk0 + nblk) are scattered into scratch,
    const S* back;              // [back0, back0 + nback) copied back from `back`
    uint64_t blk0, nblk, back0, nback;
    int N, P, w;                // register width, plane bits (2N), low bits
    RegArg a, b, c;
    int nruns;                  // the block's qubits as runs of consecutive ones, ascending
    uint8_t run_lo[34], run_len[34];
};

// Index of the first amplitude of block p: the runs' bits inserted as zeros.
template <class S>
__device__ __forceinline__ uint64_t block_base(const ArithArgs<S>& a, uint64_t p) {
    for (int j = 0; j < a.nruns; ++j) {
        const uint64_t low = p & ((1ull << a.run_lo[j]) - 1ull);
        p = ((p >> a.run_lo[j]) << (a.run_lo[j] + a.run_len[j])) | low;
    }
    return p;
}

// Offset of block value e in the state: the c register holds y's low N bits,
// the a register its high N bits.
template <class S>
__device__ __forceinline__ uint64_t block_offset(const ArithArgs<S>& a, uint32_t e) {
    const uint32_t mask = (1u << a.N) - 1u, l = e & ((1u << a.w) - 1u), y = e >> a.w;
    return l | reg_put(a.c, a.N, y & mask) | reg_put(a.a, a.N, y >> a.N);
}

// Bytes of a batch of blocks, and block values of one CTA pass.  Two batches of
// 16 MB (one scattered, one copied back) stay in L2: nine-qubit registers at
// n = 28 with batches of 8, 16, 32, 64 MB: 4.4, 3.7, 4.3, 5.4 ms.  A block above
// that is a batch of its own: whole lines count for more than L2 (complex128 at
// n = 30, a and c from qubit 10 on: ten-qubit registers, blocks of eight planes,
// 128 MB, 38.7 ms, of one plane 78.0; nine-qubit ones from qubit 3 on, 32 MB,
// 12.8 and, of four planes, 16.5 ms).
constexpr uint64_t kBatch = 1ull << 24;
constexpr int kChunk = 1024;

// A chunk of a batch scattered into the scratch buffer, each amplitude to the
// place of its image ...  The state is read in order; the scattered writes stay
// within the block's part of the buffer, 16 bytes each but complete in L2.
// (The reverse, a gather of the preimages, scatters its reads over the block's
// places in the state, 512 runs 4 MB apart for nine-qubit registers a b c, and
// read DRAM four times over: 6.6 ms for the gather alone.)
template <class S>
__device__ __forceinline__ void scatter_chunk(const ArithArgs<S>& a, uint64_t k) {
    constexpr int kAtOnce = kChunk / 256;   // independent loads in flight a thread
    const int bits = a.P + a.w;
    const uint32_t emask = (1u << bits) - 1u, mask = (1u << a.N) - 1u, wmask = (1u << a.w) - 1u;
    const uint64_t e0 = k * kChunk;
    const uint64_t base = block_base(a, a.blk0 + (e0 >> bits));
    S* const out = a.scratch + (e0 & ~(uint64_t)emask);
    S v[kAtOnce];
#pragma unroll
    for (int j = 0; j < kAtOnce; ++j)
        v[j] = a.x[base | block_offset(a, (uint32_t)(e0 + 256 * j + threadIdx.x) & emask)];
#pragma unroll
    for (int j = 0; j < kAtOnce; ++j) {
        const uint32_t e = (uint32_t)(e0 + 256 * j + threadIdx.x) & emask, l = e & wmask, y = e >> a.w;
        const uint32_t bv = reg_get(a.b, a.N, base | l);
        uint32_t av = y >> a.N, cv = y & mask;
        image(a.N, av, bv, cv);
        out[((cv | (av << a.N)) << a.w) | l] = v[j];
    }
}

// ... and a chunk copied back to its places in the state.
template <class S>
__device__ __forceinline__ void copy_back_chunk(const ArithArgs<S>& a, uint64_t k) {
    const int bits = a.P + a.w;
    const uint32_t emask = (1u << bits) - 1u;
    const uint64_t e0 = k * kChunk;
    const uint64_t base = block_base(a, a.back0 + (e0 >> bits));
    S v[kChunk / 256];
#pragma unroll
    for (int j = 0; j < kChunk / 256; ++j) v[j] = a.back[e0 + 256 * j + threadIdx.x];
#pragma unroll
    for (int j = 0; j < kChunk / 256; ++j)
        a.x[base | block_offset(a, (uint32_t)(e0 + 256 * j + threadIdx.x) & emask)] = v[j];
}

// One launch copies a batch back and scatters the next one (other blocks, the
// other half of the buffer): half as many launches, reads and writes mixed.
template <class S>
__global__ void __launch_bounds__(256) k_arith_batch(const __grid_constant__ ArithArgs<S> a) {
    const uint64_t backs = (a.nback << (a.P + a.w)) / kChunk, scatters = (a.nblk << (a.P + a.w)) / kChunk;
    const uint64_t both = backs < scatters ? backs : scatters, all = backs + scatters;
    for (uint64_t k = blockIdx.x; k < all; k += gridDim.x) {
        // alternately while both last, then what is left of either
        const bool back = k < 2 * both ? (k & 1) : backs > scatters;
        const uint64_t i = k < 2 * both ? k >> 1 : k - both;
        if (back) copy_back_chunk(a, i);
        else scatter_chunk(a, i);
    }
}

RegArg make_reg(int N, const int* q) {
    RegArg r{};
    r.lo = q[0];
    r.contiguous = 1;
    for (int j = 0; j < N; ++j) {
        r.q[j] = (uint8_t)q[j];
        if (q[j] != q[0] + j) r.contiguous = 0;
    }
    return r;
}

template <class S, int OP>
void arith_tiles(qe_state* s, int N, const int* qa, const int* qb, const int* qc, int P, const char* tag) {
    static thread_local TileArgs<S> a;
    std::memset(&a, 0, sizeof(a));
    a.x = reinterpret_cast<S*>(s->d);
    a.N = N;
    a.a = make_reg(N, qa);
    a.b = make_reg(N, qb);
    // the tile's bits: the plane's qubits and the lowest others, 64 KB in all
    // (less on small states, for at least 256 tiles).  Where a plane of 64 KB would
    // fill a tile and leaves two qubits or more below it, twice that: whole sectors
    // instead of 16 bytes (division of six-qubit complex128 registers at n = 26 from
    // qubits 2, 3, 6 on 753, 1117, 1262 us in tiles of 64 KB, 661, 946, 1176 by planes
    // one at a time, 617, 640, 689 so; from 0 and 1 on 457 and 540, 604 and 601 so)
    int below = s->n;
    for (int j = 0; j < N; ++j) below = std::min(below, OP == kDiv ? std::min(qa[j], qc[j]) : qc[j]);
    const bool wide = sizeof(S) << P == 64 * 1024 && below >= 2;
    a.T = wide ? std::min(P + 1, std::max(P, s->n - 8)) : std::min(s->n, std::max({P, std::min(sizeof(S) == 16 ? 12 : 13, s->n - 8), 5}));
    bool local[64] = {};
    for (int j = 0; j < N; ++j) {
        local[qc[j]] = true;
        if (OP == kDiv) local[qa[j]] = true;
    }
    for (int q = 0, left = a.T - P; left > 0; ++q)
        if (!local[q]) {
            local[q] = true;
            --left;
        }
    while (a.L < a.T && local[a.L]) ++a.L;
    int pos[64];
    for (int q = 0; q < s->n; ++q) {
        pos[q] = q < a.L ? q : a.L + a.kh;
        if (q >= a.L && local[q]) a.hq[a.kh++] = (uint8_t)q;
    }
    int lc[16], la[16];
    for (int j = 0; j < N; ++j) {
        lc[j] = pos[qc[j]];
        la[j] = pos[qa[j]];
    }
    a.lc = make_reg(N, lc);
    if (OP == kDiv) a.la = make_reg(N, la);
    a.ntiles = 1ull << (s->n - a.T);
    const size_t smem = sizeof(S) << a.T;
    const int threads = wide ? kWideThreads : kArithThreads;
    auto fn = wide ? k_arith_plane<S, OP, kWideThreads> : k_arith_plane<S, OP, kArithThreads>;
    QE_CUDA(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    int occ = 0;
    QE_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, fn, threads, smem));
    const uint64_t grid = std::min<uint64_t>(a.ntiles, (uint64_t)num_sms() * std::max(occ, 1));
    Launch L(s, tag, 2.0 * dim(s) * amp_bytes(s));
    fn<<<(unsigned)grid, threads, smem, s->stream>>>(a);
    QE_CUDA(cudaGetLastError());
}

template <class S>
void div_batches(qe_state* s, int N, const int* qa, const int* qb, const int* qc) {
    const int P = 2 * N;
    const size_t plane_bytes = sizeof(S) << P;
    static thread_local ArithArgs<S> a;
    std::memset(&a, 0, sizeof(a));
    a.x = reinterpret_cast<S*>(s->d);
    a.N = N;
    a.P = P;
    a.a = make_reg(N, qa);
    a.b = make_reg(N, qb);
    a.c = make_reg(N, qc);
    int bq[35], nq = 0;
    for (int j = 0; j < N; ++j) bq[nq++] = qc[j];
    for (int j = 0; j < N; ++j) bq[nq++] = qa[j];
    a.w = std::min(3, *std::min_element(bq, bq + nq));
    for (int q = 0; q < a.w; ++q) bq[nq++] = q;
    std::sort(bq, bq + nq);
    for (int j = 0; j < nq; ++j)
        if (a.nruns && bq[j] == a.run_lo[a.nruns - 1] + a.run_len[a.nruns - 1]) {
            ++a.run_len[a.nruns - 1];
        } else {
            a.run_lo[a.nruns] = (uint8_t)bq[j];
            a.run_len[a.nruns++] = 1;
        }
    const uint64_t blocks = 1ull << (s->n - P - a.w);
    const size_t block_bytes = plane_bytes << a.w;
    // batches of whole blocks through the two halves of a scratch buffer
    const uint64_t per_batch = std::max<uint64_t>(1, std::min<uint64_t>(blocks, kBatch / block_bytes));
    S* const scratch = reinterpret_cast<S*>(ensure_scratch(s, (blocks > per_batch ? 2 : 1) * per_batch * block_bytes));
    int half = 0;
    for (uint64_t p0 = 0; p0 < blocks || a.nblk; p0 += per_batch) {
        a.back = a.scratch;
        a.back0 = a.blk0;
        a.nback = a.nblk;
        a.scratch = scratch + (half ? per_batch << (P + a.w) : 0);
        half ^= 1;
        a.blk0 = p0;
        a.nblk = p0 < blocks ? std::min<uint64_t>(per_batch, blocks - p0) : 0;
        const uint64_t total = (a.nblk + a.nback) << (P + a.w);
        const unsigned grid = (unsigned)std::min<uint64_t>(total / kChunk, (uint64_t)num_sms() * 8);
        Launch L(s, "div_emulated", 1.0 * (double)total * amp_bytes(s), false);
        k_arith_batch<S><<<grid, 256, 0, s->stream>>>(a);
        QE_CUDA(cudaGetLastError());
    }
    s->stats.passes += 2;   // two full passes in total over the batches
}

}  // namespace

void launch_mul(qe_state* s, int N, const int* qa, const int* qb, const int* qc) {
    if (s->dtype == QE_C128) arith_tiles<double2, kMul>(s, N, qa, qb, qc, N, "mul_emulated");
    else arith_tiles<float2, kMul>(s, N, qa, qb, qc, N, "mul_emulated");
}

void launch_div(qe_state* s, int N, const int* qa, const int* qb, const int* qc) {
    if (((size_t)amp_bytes(s) << 2 * N) <= 64 * 1024) {
        if (s->dtype == QE_C128) arith_tiles<double2, kDiv>(s, N, qa, qb, qc, 2 * N, "div_emulated");
        else arith_tiles<float2, kDiv>(s, N, qa, qb, qc, 2 * N, "div_emulated");
    } else if (s->dtype == QE_C128) {
        div_batches<double2>(s, N, qa, qb, qc);
    } else {
        div_batches<float2>(s, N, qa, qb, qc);
    }
}

}  // namespace qe
