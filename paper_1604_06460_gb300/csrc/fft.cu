// Emulated QFT (Sec. III-B): the QFT of a register [lo, lo+m) equals, for
// every assignment of the other qubits, the length-2^m discrete Fourier
// transform with kernel exp(+2 pi i k l / 2^m) and scale 2^{-m/2}.  The
// emulator computes it as an in-place FFT instead of m(m+1)/2 gates.
//
// Three decompositions, all from the top register bits down (decimation in
// frequency) with one reversal at the end: digits of up to five qubits on the tensor
// cores (complex128, qft_tc; qft_on_tensor_cores says where), passes of up to 12
// radix-2 stages in registers four at a time (complex64 registers of several
// passes, k_fft4), and radix-2 passes in shared memory:
//
// Radix-2^r passes.  A pass loads tiles that hold whole groups of
// 2^r elements strided along its r bits into shared memory, runs r radix-2
// DIF stages there, multiplies every element by the inter-pass twiddle
// exp(s 2 pi i j2 k1 / 2^(b0+r)) (j2: the register bits below the pass, k1:
// the pass's output digit), and writes the tile back in place.  After the
// last pass the register holds the transform in bit-reversed order; a
// separate in-place tiled pass reverses it.  A register that fits in one
// tile is transformed in a single pass with the reversal done in shared
// memory.  Twiddles come from two tables of FP64-generated roots (fine and
// coarse, 2^ceil(m/2) + 2^floor(m/2) entries) stored in the policy's type.
#include <algorithm>
#include <cmath>
#include <map>
#include <type_traits>

#include "qe_arith.cuh"
#include "qe_internal.h"

namespace qe {

namespace {

constexpr int kFftThreads = 256;

template <class P>
__global__ void k_twiddles(typename P::M* fine, typename P::M* coarse, int m, int h, int sign) {
    const uint64_t nf = 1ull << h, nc = 1ull << (m - h);
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < nf + nc;
         i += (uint64_t)gridDim.x * blockDim.x) {
        const uint64_t e = i < nf ? i : ((i - nf) << h);
        // exp(sign * 2 pi i e / 2^m): the angle in units of pi is exact
        const double x = scalbn((double)e, 1 - m);
        double sn, cs;
        sincospi(x, &sn, &cs);
        typename P::M w = P::from_d(cs, sign > 0 ? sn : -sn);
        if (i < nf) fine[i] = w;
        else coarse[i - nf] = w;
    }
}

template <class P>
struct FftArgs {
    typename P::S* x;
    const typename P::M* fine;
    const typename P::M* coarse;
    uint64_t ntiles;
    int L, T, kh;
    uint8_t hq[16];
    int P0;       // tile-local position of the lowest pass bit
    int r;        // bits in this pass
    int b0;       // lowest register bit of this pass (register-relative)
    int lo, m, h; // register placement, size, fine-table bits
    int twiddle;  // multiply by the inter-pass twiddle
    int natural;  // single pass: undo the bit reversal inside the tile
    int scale_on;
    int gmax;     // radix-2 stages per register group (1..4)
    typename P::M scale;
};

template <class P>
__device__ __forceinline__ typename P::M root(const FftArgs<P>& a, uint64_t e) {
    return P::cmul(a.coarse[e >> a.h], a.fine[e & ((1ull << a.h) - 1ull)]);
}

// Asynchronous global -> shared copy of one amplitude (cp.async, 16 or 8 bytes).
template <class S>
__device__ __forceinline__ void async_copy(void* dst, const S* src) {
    const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
    if (sizeof(S) == 16)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(src));
    else
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(d), "l"(src));
}
__device__ __forceinline__ void async_commit() { asm volatile("cp.async.commit_group;"); }
__device__ __forceinline__ void async_wait_prev() { asm volatile("cp.async.wait_group 1;" ::: "memory"); }

// Shared-memory slot of tile element i: one pad slot per 16 elements, so that
// the 16-element stride of the lowest register group maps lanes to distinct
// banks.
__device__ __forceinline__ uint32_t pad16(uint32_t i) { return i + (i >> 4); }

// G radix-2 DIF stages s_hi, s_hi-1, ..., s_hi-G+1 of the tile's groups, in
// registers.  Element j (G bits) of a thread's set sits at local index
// base | (j << (P0 + s_lo)); its in-group index is gp = (local >> P0) & (R-1)
// and stage s multiplies the difference by roots[2^s - 1 + (gp mod 2^s)].
template <class P, int G>
__device__ __forceinline__ void stage_group(typename P::V* tile, const typename P::M* roots, int Tn, int P0,
                                            int s_hi) {
    using V = typename P::V;
    constexpr int E = 1 << G;
    const int s_lo = s_hi - G + 1;
    const int sh = P0 + s_lo;
    const uint32_t below = (1u << sh) - 1u;
    const int nbase = Tn >> G;
    for (int b = threadIdx.x; b < nbase; b += blockDim.x) {
        const uint32_t base = (((uint32_t)b & ~below) << G) | ((uint32_t)b & below);
        V v[E];
#pragma unroll
        for (int j = 0; j < E; ++j) v[j] = tile[pad16(base | ((uint32_t)j << sh))];
        const uint32_t gp0 = base >> P0;   // the thread's fixed in-group bits (group bits zero)
#pragma unroll
        for (int t = G - 1; t >= 0; --t) {
            const int s = s_lo + t;
            const uint32_t smask = (1u << s) - 1u;
#pragma unroll
            for (int j = 0; j < E; ++j) {
                if (j & (1 << t)) continue;
                const int j2 = j | (1 << t);
                const uint32_t p = (gp0 | ((uint32_t)j << s_lo)) & smask;
                const typename P::M w = roots[(1u << s) - 1u + p];
                const V u = v[j], x = v[j2];
                v[j] = P::add(u, x);
                v[j2] = P::cmul(w, P::sub(u, x));
            }
        }
#pragma unroll
        for (int j = 0; j < E; ++j) tile[pad16(base | ((uint32_t)j << sh))] = v[j];
    }
}

template <class P>
__global__ void __launch_bounds__(kFftThreads) k_fft_pass(const __grid_constant__ FftArgs<P> a) {
    using V = typename P::V;
    using M = typename P::M;
    using S = typename P::S;
    static_assert(sizeof(V) == sizeof(S), "tile slots hold the raw amplitude before conversion");
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int Tn = 1 << a.T;
    const int slots = Tn + Tn / 16;
    // two tiles: the next one is copied asynchronously while the current one is transformed
    V* buf[2] = {reinterpret_cast<V*>(smem_raw), reinterpret_cast<V*>(smem_raw) + slots};
    M* roots = reinterpret_cast<M*>(buf[1] + slots);
    __shared__ uint64_t offA[64], offB[64];
    const int tid = threadIdx.x, nth = blockDim.x;
    const int R = 1 << a.r;
    // per-stage tables: roots[2^s - 1 + p] = exp(sign 2 pi i p / 2^(s+1)), p < 2^s,
    // so that lanes with consecutive p read consecutive entries
    for (int e = tid; e < R - 1; e += nth) {
        const int s = 31 - __clz(e + 1);
        const uint64_t p = (uint64_t)(e + 1 - (1 << s));
        roots[e] = root(a, p << (a.m - s - 1));
    }
    if (tid < 64) {
        uint64_t oa = 0, ob = 0;
        for (int j = 0; j < 6 && j < a.kh; ++j)
            if ((tid >> j) & 1) oa |= 1ull << a.hq[j];
        for (int j = 6; j < a.kh; ++j)
            if ((tid >> (j - 6)) & 1) ob |= 1ull << a.hq[j];
        offA[tid] = oa;
        offB[tid] = ob;
    }
    __syncthreads();
    const uint32_t lowmask = (1u << a.L) - 1u;
    const uint64_t j2mask = (1ull << a.b0) - 1ull;
    const uint64_t emask = (1ull << (a.b0 + a.r)) - 1ull;
    auto issue = [&](uint64_t t, V* dst) {
        const uint64_t base = insert_zero_bits(t << a.L, a.hq, a.kh);
        for (int i = tid; i < Tn; i += nth) {
            const uint32_t hi = (uint32_t)i >> a.L;
            async_copy<S>(dst + pad16(i), a.x + base + (i & lowmask) + offA[hi & 63] + offB[hi >> 6]);
        }
    };
    uint64_t t = blockIdx.x;
    if (t < a.ntiles) issue(t, buf[0]);
    async_commit();
    for (int it = 0; t < a.ntiles; t += gridDim.x, ++it) {
        V* tile = buf[it & 1];
        const uint64_t tn = t + gridDim.x;
        if (tn < a.ntiles) issue(tn, buf[(it + 1) & 1]);
        async_commit();
        async_wait_prev();
        __syncthreads();
        if (sizeof(S) == 16 && !std::is_same<V, S>::value) {
            // raw amplitudes -> the policy's working type, in place
            for (int i = tid; i < Tn; i += nth) {
                const S raw = *reinterpret_cast<const S*>(tile + pad16(i));
                tile[pad16(i)] = P::load(raw);
            }
            __syncthreads();
        }
        const uint64_t base = insert_zero_bits(t << a.L, a.hq, a.kh);
        // radix-2 DIF stages from the top pass bit down, a few at a time in
        // registers: a thread owns the 2^g elements that differ in the g bits
        // of the group, so each group costs one shared-memory round trip
        for (int s_hi = a.r - 1; s_hi >= 0; s_hi -= a.gmax) {
            const int g = s_hi + 1 < a.gmax ? s_hi + 1 : a.gmax;
            switch (g) {
                case 4: stage_group<P, 4>(tile, roots, Tn, a.P0, s_hi); break;
                case 3: stage_group<P, 3>(tile, roots, Tn, a.P0, s_hi); break;
                case 2: stage_group<P, 2>(tile, roots, Tn, a.P0, s_hi); break;
                default: stage_group<P, 1>(tile, roots, Tn, a.P0, s_hi); break;
            }
            __syncthreads();
        }
        for (int i = tid; i < Tn; i += nth) {
            const uint32_t hi = (uint32_t)i >> a.L;
            const uint64_t G = base + (i & lowmask) + offA[hi & 63] + offB[hi >> 6];
            const uint32_t gp = ((uint32_t)i >> a.P0) & (uint32_t)(R - 1);
            const uint32_t rev = (a.r > 0) ? (__brev(gp) >> (32 - a.r)) : 0u;
            V v;
            if (a.natural) {
                // position gp receives the element whose in-group index is rev(gp)
                const uint32_t src = ((uint32_t)i & ~((uint32_t)(R - 1) << a.P0)) | (rev << a.P0);
                v = tile[pad16(src)];
            } else {
                v = tile[pad16(i)];
            }
            if (a.twiddle) {
                const uint64_t j2 = (G >> a.lo) & j2mask;
                const uint64_t e = ((j2 * (uint64_t)rev) & emask) << (a.m - a.b0 - a.r);
                v = P::cmul(root(a, e), v);
            }
            if (a.scale_on) v = P::cmul(a.scale, v);
            a.x[G] = P::store(v);
        }
        __syncthreads();
    }
    async_wait_prev();
}

// --------------------------------------------------------------- bitrev
// In-place reversal of the register value's bits.  Work item = (outer bits,
// middle value Mv <= rev(Mv)); tiles X(Mv) and Y(rev Mv) hold elements
// [b][a][w] (b: top c register bits, a: bottom c register bits, w: the lo
// qubits below the register) and are exchanged transposed and bit-reversed.
template <class S>
struct RevArgs {
    S* x;
    uint64_t items;
    int lo, m, c;
};

__device__ __forceinline__ uint64_t bit_rev(uint64_t v, int bits) { return bits > 0 ? (__brevll(v) >> (64 - bits)) : 0ull; }

constexpr int kRevThreads = 256;
// Tile bits: 32 KB a tile.  n = 30 complex128 9.0 -> 8.8 ms and n = 27 complex64
// 0.73 -> 0.52 ms (0.32 for one pass) with shifts for divisions, loads in
// batches of eight, the swizzle below and, for 8-byte elements, one bit more;
// tiles of 64 KB measured 8.96 ms, one tile with the other in registers 8.4 ms
// but 0.66 ms in complex64.  Rows of 512 bytes bound it: with rows of 1 KB
// (one qubit below the register) n = 27 takes 0.89 instead of 1.11 ms.
template <class S>
constexpr int kRevBits = sizeof(S) == 16 ? 11 : 12;

template <class S>
__global__ void __launch_bounds__(kRevThreads) k_bitrev(const __grid_constant__ RevArgs<S> a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    constexpr int kAtOnce = 8;   // independent loads in flight a thread
    const int c = a.c, ab = c + a.lo;                 // bits of a row (a, w)
    const uint32_t n = 1u << (c + ab), amask = (1u << ab) - 1u, wmask = (1u << a.lo) - 1u;
    S* const X = reinterpret_cast<S*>(smem_raw);
    S* const Y = X + n;
    // Tile slot (row, place in the row).  The lanes that one phase of an access
    // serves (8 of 16 bytes, 16 of 8) read the low bits of a, hence rows that
    // differ in their top bits: those are XORed into the place, above the w bits
    // that vary along with them.
    constexpr int kPhase = sizeof(S) == 16 ? 3 : 4;
    const int k = max(0, min(c, kPhase - a.lo));
    auto slot = [&](uint32_t r, uint32_t place) { return (r << ab) | (place ^ (k ? (r >> (c - k)) << a.lo : 0u)); };
    const int mid_bits = a.m - 2 * c;
    const uint64_t nmid = 1ull << mid_bits;
    const int shb = a.lo + a.m - c;
    for (uint64_t item = blockIdx.x; item < a.items; item += gridDim.x) {
        const uint64_t mv = item & (nmid - 1ull);
        const uint64_t outer = item >> mid_bits;
        const uint64_t mr = bit_rev(mv, mid_bits);
        if (mv > mr) continue;
        const bool self = (mv == mr);
        const uint64_t obase = outer << (a.lo + a.m);
        S* const bx = a.x + (obase | (mv << (a.lo + c)));
        S* const by = a.x + (obase | (mr << (a.lo + c)));
        auto off = [&](uint32_t i) { return ((uint64_t)(i >> ab) << shb) | (i & amask); };
        for (uint32_t i0 = threadIdx.x; i0 < n; i0 += kRevThreads * kAtOnce) {
            S vx[kAtOnce], vy[kAtOnce];
#pragma unroll
            for (int u = 0; u < kAtOnce; ++u) {
                const uint32_t i = i0 + kRevThreads * u;
                if (i < n) {
                    vx[u] = bx[off(i)];
                    if (!self) vy[u] = by[off(i)];
                }
            }
#pragma unroll
            for (int u = 0; u < kAtOnce; ++u) {
                const uint32_t i = i0 + kRevThreads * u;
                if (i < n) {
                    X[slot(i >> ab, i & amask)] = vx[u];
                    if (!self) Y[slot(i >> ab, i & amask)] = vy[u];
                }
            }
        }
        __syncthreads();
        const S* srcX = self ? X : Y;   // destination tile X(mv) receives from Y
#pragma unroll 4
        for (uint32_t i = threadIdx.x; i < n; i += kRevThreads) {
            const uint32_t b2 = i >> ab, a2 = (i & amask) >> a.lo, w = i & wmask;
            const uint32_t rb = (uint32_t)bit_rev(a2, c);   // source b
            const uint32_t ra = (uint32_t)bit_rev(b2, c);   // source a
            const uint32_t src = slot(rb, (ra << a.lo) | w);
            bx[off(i)] = srcX[src];
            if (!self) by[off(i)] = X[src];
        }
        __syncthreads();
    }
}

struct TableKey {
    int m, sign, policy;
    bool operator<(const TableKey& o) const {
        return m != o.m ? m < o.m : sign != o.sign ? sign < o.sign : policy < o.policy;
    }
};
struct Table {
    void* fine = nullptr;
    void* coarse = nullptr;
};
std::map<std::pair<int, TableKey>, Table> g_tables;   // (device, key) -> table

template <class P>
Table get_tables(qe_state* s, int m, int sign, int pol) {
    int dev = 0;
    QE_CUDA(cudaGetDevice(&dev));
    auto key = std::make_pair(dev, TableKey{m, sign, pol});
    auto it = g_tables.find(key);
    if (it != g_tables.end()) return it->second;
    const int h = (m + 1) / 2;
    Table t;
    QE_CUDA(cudaMalloc(&t.fine, sizeof(typename P::M) << h));
    QE_CUDA(cudaMalloc(&t.coarse, sizeof(typename P::M) << (m - h)));
    uint64_t total = (1ull << h) + (1ull << (m - h));
    unsigned grid = (unsigned)std::min<uint64_t>((total + 255) / 256, 4096);
    Launch L(s, "fft_twiddles", 0.0, false);
    k_twiddles<P><<<grid, 256, 0, s->stream>>>((typename P::M*)t.fine, (typename P::M*)t.coarse, m, h, sign);
    QE_CUDA(cudaGetLastError());
    g_tables[key] = t;
    return t;
}

struct Geom {
    int T = 0, L = 0, kh = 0;
    uint8_t hq[16] = {0};
};
// Tile of at most 2^Tt elements containing the register bits [g0, g0+r).
Geom pass_geom(int n, int g0, int r, int Tt) {
    Tt = std::min(Tt, n);
    for (int L = Tt; L >= 0; --L) {
        int kh = 0;
        for (int q = g0; q < g0 + r; ++q) kh += q >= L;
        if (L + kh <= Tt) {
            Geom g;
            g.L = L;
            g.kh = kh;
            g.T = L + kh;
            int j = 0;
            for (int q = g0; q < g0 + r; ++q)
                if (q >= L) g.hq[j++] = (uint8_t)q;
            return g;
        }
    }
    fail(QE_ERR_ARG, "no FFT tile geometry");
}

template <class P>
void fft_impl(qe_state* s, int lo, int m, int inverse, int pol) {
    const int sign = inverse ? -1 : 1;
    Table tb = get_tables<P>(s, m, sign, pol);
    const int Tmax = (sizeof(typename P::V) >= 16) ? 11 : 12;
    const int Lmin = 3;   // runs of >= 8 amplitudes (measured best: fewer passes outweigh shorter runs)
    const int rb_max = Tmax - std::min(lo, Lmin);
    std::vector<std::pair<int, int>> passes;   // (b0, r), top first
    if (m <= rb_max) {
        passes.push_back({0, m});
    } else {
        const int ru_max = Tmax - Lmin;
        const int rest = m - rb_max;
        const int nup = (rest + ru_max - 1) / ru_max;
        int top = m;
        for (int p = 0; p < nup; ++p) {
            int r = rest / nup + (p < rest % nup ? 1 : 0);
            passes.push_back({top - r, r});
            top -= r;
        }
        passes.push_back({0, top});
    }
    static thread_local FftArgs<P> a;
    a.x = reinterpret_cast<typename P::S*>(s->d);
    a.fine = (const typename P::M*)tb.fine;
    a.coarse = (const typename P::M*)tb.coarse;
    a.lo = lo;
    a.m = m;
    a.h = (m + 1) / 2;
    const double scale = std::pow(2.0, -0.5 * m);
    a.scale = P::mat(scale, 0.0);
    const bool single = passes.size() == 1;
    for (size_t p = 0; p < passes.size(); ++p) {
        const int b0 = passes[p].first, r = passes[p].second;
        Geom g = pass_geom(s->n, lo + b0, r, Tmax);
        a.L = g.L;
        a.T = g.T;
        a.kh = g.kh;
        for (int j = 0; j < 16; ++j) a.hq[j] = g.hq[j];
        a.P0 = std::min(lo + b0, g.L);
        a.r = r;
        a.b0 = b0;
        a.ntiles = 1ull << (s->n - g.T);
        a.twiddle = b0 > 0;
        a.natural = single;
        a.scale_on = (p + 1 == passes.size());
        size_t smem = 2 * sizeof(typename P::V) * (((size_t)1 << g.T) + ((size_t)1 << g.T) / 16) +
                      sizeof(typename P::M) * ((size_t)1 << r);
        // three radix-2 stages per register group and 256 threads measured
        // fastest on GB300 for both complex64 and complex128 tiles
        a.gmax = 3;
        const int threads = std::max(64, std::min(256, (1 << g.T) >> a.gmax));
        auto fn = k_fft_pass<P>;
        QE_CUDA(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        int occ = 0;
        QE_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, fn, threads, smem));
        uint64_t grid = std::min<uint64_t>(a.ntiles, (uint64_t)num_sms() * std::max(occ, 1));
        Launch L(s, "fft_pass", 2.0 * dim(s) * amp_bytes(s));
        fn<<<(unsigned)grid, threads, smem, s->stream>>>(a);
        QE_CUDA(cudaGetLastError());
    }
    if (!single) launch_bitrev(s, lo, m);
}

template <class S>
__global__ void __launch_bounds__(256) k_bitrev_chunks(S* __restrict__ x, uint64_t count, int lo, int m) {
    const uint64_t rmask = ((1ull << m) - 1ull) << lo;
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < count;
         i += (uint64_t)gridDim.x * blockDim.x) {
        const uint64_t k = (i & rmask) >> lo;
        const uint64_t kr = bit_rev(k, m);
        if (k < kr) {
            const uint64_t j = (i & ~rmask) | (kr << lo);
            S t = x[i];
            x[i] = x[j];
            x[j] = t;
        }
    }
}

// Registers whose slices of 2^(lo + m) amplitudes fit a tile: tiles of 2^kRevBits
// contiguous amplitudes, permuted through shared memory (exchanges of their
// small end blocks moved pieces of a few lines: six qubits from 0 on at n = 26
// 3.0 -> 0.37 ms).  The lanes of a phase read places whose varying bits are
// consecutive; every bit above the lowest three (four for 8 bytes) is XORed into
// one of those, consecutive ones into different ones.
template <class S>
__global__ void __launch_bounds__(kRevThreads) k_bitrev_slices(S* __restrict__ x, uint64_t tiles, int T, int lo, int m) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    S* const buf = reinterpret_cast<S*>(smem_raw);
    constexpr int kFold = sizeof(S) == 16 ? 3 : 4;
    auto slot = [&](uint32_t i) {
        uint32_t f = 0;
#pragma unroll
        for (int b = kFold; b < kRevBits<S>; b += kFold) f ^= i >> b;
        return i ^ (f & ((1u << kFold) - 1u));
    };
    const uint32_t rmask = ((1u << m) - 1u) << lo, n = 1u << T;
    for (uint64_t t = blockIdx.x; t < tiles; t += gridDim.x) {
        S* const xt = x + (t << T);
#pragma unroll 8
        for (uint32_t i = threadIdx.x; i < n; i += kRevThreads) buf[slot(i)] = xt[i];
        __syncthreads();
#pragma unroll 8
        for (uint32_t i = threadIdx.x; i < n; i += kRevThreads)
            xt[i] = buf[slot((i & ~rmask) | ((uint32_t)bit_rev((i & rmask) >> lo, m) << lo))];
        __syncthreads();
    }
}

template <class P>
void bitrev_impl(qe_state* s, int lo, int m, const char* tag = "bitrev") {
    if (m <= 1) return;
    using S = typename P::S;
    Launch L(s, tag, 2.0 * dim(s) * amp_bytes(s));
    // end blocks of c bits (2c <= m) in tiles of 2^(2c + lo) <= 2^kRevBits
    const int c = std::min(m / 2, std::max(0, (kRevBits<S> - lo) / 2));
    if (lo + m <= kRevBits<S>) {
        const int T = std::min(s->n, kRevBits<S>);
        const uint64_t tiles = 1ull << (s->n - T);
        const size_t smem = sizeof(S) << T;
        int occ = 0;
        QE_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_bitrev_slices<S>, kRevThreads, smem));
        const uint64_t grid = std::min<uint64_t>(tiles, (uint64_t)num_sms() * std::max(occ, 1));
        k_bitrev_slices<S><<<(unsigned)grid, kRevThreads, smem, s->stream>>>(reinterpret_cast<S*>(s->d), tiles, T, lo, m);
    } else if (lo >= 5 || c == 0) {
        // chunks of >= 32 contiguous amplitudes move as units: coalesced pair swaps
        const uint64_t count = dim(s);
        unsigned grid = (unsigned)std::min<uint64_t>((count + 255) / 256, (uint64_t)num_sms() * 8);
        k_bitrev_chunks<S><<<grid, 256, 0, s->stream>>>(reinterpret_cast<S*>(s->d), count, lo, m);
    } else {
        RevArgs<S> a;
        a.x = reinterpret_cast<S*>(s->d);
        a.lo = lo;
        a.m = m;
        a.c = c;
        a.items = (1ull << (s->n - lo - m)) << (m - 2 * a.c);
        const size_t smem = sizeof(S) * 2 << (2 * c + lo);
        auto fn = k_bitrev<S>;
        QE_CUDA(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        int occ = 0;
        QE_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, fn, kRevThreads, smem));
        uint64_t grid = std::min<uint64_t>(a.items, (uint64_t)num_sms() * std::max(occ, 1));
        fn<<<(unsigned)grid, kRevThreads, smem, s->stream>>>(a);
    }
    QE_CUDA(cudaGetLastError());
}

// ------------------------------------------------ complex64, several passes
// A pass over r = 5..12 register bits of a complex64 state, in tiles of 2^12
// amplitudes: the bits in two or three groups of 2..4, each a 2^g-point
// transform in registers whose roots are constants, a twiddle from a shared
// table between groups, the tile in shared memory only between groups (the
// first reads global memory, the last writes it).  The inter-pass twiddles are
// computed: the angle k' l / 2^M is an exact 32-bit fraction of a turn, so a
// root costs one sincospif of at most pi/4 and no table in memory; a thread's
// 2^g outputs share one (A) and take the powers of another (B): with
// k = 4a + b, w_k = (A B^(4a)) B^b, products of two rounded roots as a two-level
// table gives.  What bounded the radix-2 passes that this replaces was their
// table reads (two 32-byte sectors an amplitude): 27 qubits at n = 27 1.09 ->
// 0.41 ms a pass (0.32 copied), with the reversal 4.10 -> 1.73 ms.
struct Fft4Args {
    float2* x;
    uint64_t ntiles;
    int L, kh;      // tile: 2^L contiguous amplitudes, kh = r (pass bits above them) or 0 (among them)
    int g0;         // qubit of the pass's lowest bit
    int P0;         // its tile-local place
    int b0;         // register bits below the pass
    int lo;
    float scale;    // of the last pass (b0 = 0)
};

using fc = unsigned long long;   // (re, im) as packed floats
__device__ __forceinline__ fc fc_pack(float x, float y) {
    fc r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(x), "f"(y));
    return r;
}
__device__ __forceinline__ float2 fc_unpack(fc a) {
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(a));
    return r;
}
__device__ __forceinline__ fc fc_add(fc a, fc b) {
    fc r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ fc fc_sub(fc a, fc b) {
    fc r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ fc fc_mul2(fc a, fc b) {
    fc r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ fc fc_cmul(fc w, fc v) {
    const float2 f = fc_unpack(w), u = fc_unpack(v);
    const fc t = fc_mul2(fc_pack(-f.y, f.y), fc_pack(u.y, u.x));
    fc r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(fc_pack(f.x, f.x)), "l"(v), "l"(t));
    return r;
}
// exp(SIGN 2 pi i th / 2^32)
template <int SIGN>
__device__ __forceinline__ fc turn(uint32_t th) {
    const uint32_t q = (th + (1u << 29)) >> 30;              // nearest quarter turn
    const float x = (float)(int)(th - (q << 30)) * 0x1p-31f;   // what is left, in units of pi
    float s, c;
    sincospif(x, &s, &c);
    const float re = (q & 1u) ? -s : c, im = (q & 1u) ? c : s;
    const bool neg = q & 2u;
    return fc_pack(neg ? -re : re, (neg != (SIGN < 0)) ? -im : im);
}
// exp(2 pi i k / 16) for k < 8
__device__ constexpr float kCos16[8] = {1.0f, 0.92387953251128674f, 0.70710678118654752f, 0.38268343236508977f,
                                        0.0f, -0.38268343236508977f, -0.70710678118654752f, -0.92387953251128674f};

// v <- the 2^G-point transform, output l at the bit-reversed place.
template <int G, int SIGN>
__device__ __forceinline__ void small_dft(fc* v) {
    constexpr int E = 1 << G;
#pragma unroll
    for (int h = E / 2; h >= 1; h /= 2)
#pragma unroll
        for (int j = 0; j < E; ++j) {
            if (j & h) continue;
            const fc u = v[j], x = v[j | h];
            v[j] = fc_add(u, x);
            const fc d = fc_sub(u, x);
            const int k = (j & (h - 1)) * (8 / h);           // root exp(SIGN 2 pi i k / 16)
            if (k == 0) {
                v[j | h] = d;
            } else if (k == 4) {
                const float2 f = fc_unpack(d);
                v[j | h] = SIGN > 0 ? fc_pack(-f.y, f.x) : fc_pack(f.y, -f.x);
            } else {
                const float sn = k < 4 ? -kCos16[k + 4] : kCos16[k - 4];     // sin(2 pi k / 16)
                v[j | h] = fc_cmul(fc_pack(kCos16[k], SIGN > 0 ? sn : -sn), d);
            }
        }
}
__host__ __device__ constexpr int rev_bits(int v, int bits) {
    int r = 0;
    for (int j = 0; j < bits; ++j) r |= ((v >> j) & 1) << (bits - 1 - j);
    return r;
}
// Conflict-free slot of a tile element or root (16 8-byte lanes a phase).
__device__ __forceinline__ uint32_t slot16(uint32_t i) { return i ^ ((i >> 4) & 15u); }

constexpr int kFft4Bits = 12, kFft4Threads = 256;

// One group: pass bits [SLO, SLO + G) of the tile at tile0 in global memory.
template <int R, int SLO, int G, int SIGN>
__device__ __forceinline__ void fft4_group(const Fft4Args& a, float2* tile0, uint32_t j2_tile, fc* tile, const fc* roots) {
    constexpr int E = 1 << G;
    constexpr bool kFirst = SLO + G == R, kLast = SLO == 0;
    const int sh = a.P0 + SLO;
    const uint32_t below = (1u << sh) - 1u, lowmask = (1u << a.L) - 1u;
#pragma unroll 1
    for (uint32_t b = threadIdx.x; b < (1u << (kFft4Bits - G)); b += kFft4Threads) {
        const uint32_t base = ((b & ~below) << G) | (b & below);
        const uint64_t at = (base & lowmask) | (a.kh ? (uint64_t)(base >> a.L) << a.g0 : (uint64_t)0);
        const uint64_t stride = 1ull << (a.g0 + SLO);
        fc v[E];
        if constexpr (kFirst) {
#pragma unroll
            for (int j = 0; j < E; ++j) v[j] = *reinterpret_cast<const fc*>(tile0 + at + j * stride);
        } else {
#pragma unroll
            for (int j = 0; j < E; ++j) v[j] = tile[slot16(base | ((uint32_t)j << sh))];
        }
        small_dft<G, SIGN>(v);
        const uint32_t gp = (base >> a.P0) & ((1u << R) - 1u);
        if constexpr (!kLast) {
            // twiddle by the pass bits below this group
            const uint32_t low = gp & ((1u << SLO) - 1u);
#pragma unroll
            for (int j = 1; j < E; ++j)
                v[j] = fc_cmul(roots[slot16((low * (uint32_t)rev_bits(j, G)) << (R - SLO - G))], v[j]);
#pragma unroll
            for (int j = 0; j < E; ++j) tile[slot16(base | ((uint32_t)j << sh))] = v[j];
        } else {
            if (a.b0 > 0) {
                // twiddle by the register bits below the pass: j2 l / 2^(b0 + R)
                const uint64_t j2 = j2_tile | ((((base & lowmask) & (a.kh ? ~0u : (1u << a.g0) - 1u)) >> a.lo));
                const uint32_t rb = __brev(gp) >> (32 - R);
                const int up = 64 - (a.b0 + R);
                const uint32_t tA = (uint32_t)(((j2 * rb) << up) >> 32), tB = (uint32_t)(((j2 << (R - G)) << up) >> 32);
                fc wb[4];
#pragma unroll
                for (int k = 1; k < 4 && k < E; ++k) wb[k] = turn<SIGN>(tB * (uint32_t)k);
#pragma unroll
                for (int ka = 0; ka < E / 4; ++ka) {
                    const fc wa = turn<SIGN>(tA + tB * (uint32_t)(4 * ka));
#pragma unroll
                    for (int kb = 0; kb < 4; ++kb) {
                        const int j = rev_bits(4 * ka + kb, G);
                        v[j] = fc_cmul(kb ? fc_cmul(wa, wb[kb]) : wa, v[j]);
                    }
                }
            } else {
                const fc sc = fc_pack(a.scale, a.scale);
#pragma unroll
                for (int j = 0; j < E; ++j) v[j] = fc_mul2(sc, v[j]);
            }
            fc* const out = reinterpret_cast<fc*>(tile0 + at);
            if (a.g0 == 0) {
                // a thread's outputs are contiguous: 32 bytes at a time
#pragma unroll
                for (int j = 0; j < E; j += 4)
                    asm volatile("st.global.v4.b64 [%0], {%1, %2, %3, %4};" ::"l"(out + j), "l"(v[j]), "l"(v[j + 1]),
                                 "l"(v[j + 2]), "l"(v[j + 3])
                                 : "memory");
            } else {
#pragma unroll
                for (int j = 0; j < E; ++j) out[j * stride] = v[j];
            }
        }
    }
}

template <int R, int SIGN>
__global__ void __launch_bounds__(kFft4Threads, 4) k_fft4(const __grid_constant__ Fft4Args a) {
    static_assert(R >= 5 && R <= 12, "two or three groups of 2..4 bits");
    extern __shared__ __align__(16) unsigned char smem_raw[];
    fc* const tile = reinterpret_cast<fc*>(smem_raw);
    fc* const roots = tile + (1 << kFft4Bits);
    constexpr int NG = R <= 8 ? 2 : 3;
    constexpr int G1 = (R + NG - 1) / NG, G2 = (R - G1 + NG - 2) / (NG - 1), G3 = R - G1 - G2;   // from the top
    for (uint32_t e = threadIdx.x; e < (1u << R); e += kFft4Threads) roots[slot16(e)] = turn<SIGN>(e << (32 - R));
    __syncthreads();
    for (uint64_t t = blockIdx.x; t < a.ntiles; t += gridDim.x) {
        // the pass bits inserted as zeros above the contiguous ones
        const uint64_t u = t << a.L;
        const uint64_t base = a.kh ? ((u >> a.g0) << (a.g0 + R)) | (u & ((1ull << a.g0) - 1ull)) : u;
        float2* const tile0 = a.x + base;
        const uint32_t j2 = (uint32_t)((base >> a.lo) & ((1ull << a.b0) - 1ull));
        fft4_group<R, R - G1, G1, SIGN>(a, tile0, j2, tile, roots);
        __syncthreads();
        if constexpr (NG == 3) {
            fft4_group<R, G3, G2, SIGN>(a, tile0, j2, tile, roots);
            __syncthreads();
            fft4_group<R, 0, G3, SIGN>(a, tile0, j2, tile, roots);
        } else {
            fft4_group<R, 0, G2, SIGN>(a, tile0, j2, tile, roots);
        }
        __syncthreads();
    }
}

template <int R>
void fft4_launch(qe_state* s, const Fft4Args& a, int sign) {
    auto fn = sign > 0 ? k_fft4<R, 1> : k_fft4<R, -1>;
    const size_t smem = sizeof(fc) * ((size_t)(1 << kFft4Bits) + ((size_t)1 << R));
    QE_CUDA(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    int occ = 0;
    QE_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, fn, kFft4Threads, smem));
    const uint64_t grid = std::min<uint64_t>(a.ntiles, (uint64_t)num_sms() * std::max(occ, 1));
    Launch L(s, "fft_pass", 2.0 * dim(s) * amp_bytes(s));
    fn<<<(unsigned)grid, kFft4Threads, smem, s->stream>>>(a);
    QE_CUDA(cudaGetLastError());
}

// Complex64 registers of more than one pass (m > 12 - min(lo, 3), hence n >= 12).
void fft4(qe_state* s, int lo, int m, int inverse) {
    const int last_max = kFft4Bits - std::min(lo, 3), up_max = kFft4Bits - 3;   // runs of at least 8 amplitudes
    const int np = 1 + (m - last_max + up_max - 1) / up_max;
    // upper passes of 8 bits (two groups of four) where that suffices
    const int up = std::max((m - last_max + np - 2) / (np - 1), std::min(8, m / np));
    Fft4Args a{};
    a.x = reinterpret_cast<float2*>(s->d);
    a.ntiles = 1ull << (s->n - kFft4Bits);
    a.lo = lo;
    a.scale = (float)std::pow(2.0, -0.5 * m);
    int top = m;
    for (int p = 0; p < np; ++p) {
        const int r = p + 1 < np ? up : top;
        top -= r;
        a.b0 = top;
        a.g0 = lo + top;
        // the pass bits within the lowest 12, or above 12 - r contiguous ones
        const bool low = a.g0 + r <= kFft4Bits;
        a.L = low ? kFft4Bits : kFft4Bits - r;
        a.kh = low ? 0 : r;
        a.P0 = low ? a.g0 : a.L;
        const int sign = inverse ? -1 : 1;
        switch (r) {
            case 5: fft4_launch<5>(s, a, sign); break;
            case 6: fft4_launch<6>(s, a, sign); break;
            case 7: fft4_launch<7>(s, a, sign); break;
            case 8: fft4_launch<8>(s, a, sign); break;
            case 9: fft4_launch<9>(s, a, sign); break;
            case 10: fft4_launch<10>(s, a, sign); break;
            case 11: fft4_launch<11>(s, a, sign); break;
            case 12: fft4_launch<12>(s, a, sign); break;
            default: fail(QE_ERR_ARG, "no FFT pass plan");
        }
    }
    launch_bitrev(s, lo, m);
}

// ------------------------------------------------ tensor-core digit passes
// The QFT of a register of m qubits as G = ceil(m / 5) dense blocks of up to five
// qubits on the tensor cores (Cooley-Tukey, digits from the top).  With the
// digits of the register value from the top k_0, k_1, ... (k = k_0 2^(m-d_0) + k')
// and the outputs so far l = l_0 + 2^(d_0) l_1 + ..., digit j is
//   y = sum_(k_j) x(k_j) 2^(-d_j/2) w_(2^(P+d_j))^(k_j (l + 2^P l_j)),
// P = d_0 + .. + d_(j-1): its 2^(d_j)-point transform with the twiddle
// w_(2^(P+d_j))^(k_j l) folded into the matrix, which then depends on the
// outputs l (qubits outside the block).  What is left of the twiddles, by the
// lower bits k' that no digit of this group will meet, is w_(2^m)^(k' l) for l
// all the outputs of the group: one diagonal pass for each group of digits
// instead of one for each digit.  Every digit leaves its output bit-reversed in
// its own qubits, so one bit reversal of the register restores the natural
// order for any split into digits (a single digit writes it directly).
//
// A digit joins the group while a matrix still serves at least 16 tiles
// (P <= n - 16: rebuilding it costs a segment of the pipeline, about two tiles)
// and its roots fit a direct table (P + d <= 20); the digits are then spread
// evenly over that number of groups where that keeps both limits.  Measured on complex128 in the FP64 mode,
// against dense blocks with a twiddle pass after each (m a multiple of its
// digit) or the shared-memory transform: the 30-qubit QFT 121 -> 79 ms (six
// digits 54, one twiddle pass 15.4, reversal 9), 29 qubits 161 -> 39.5 ms, 17
// qubits from qubit 5 of 27 on 24.9 -> 5.9 ms.
struct TwArgs {
    double2* x;
    const double2* fine;
    const double2* coarse;
    const double2* direct;   // w_(2^(base + S))^j for all j, when that order is at most 2^20 (else null)
    uint64_t count;
    int lo, h;
    int base, S;  // the group just transformed: register bits [base, base + S)
    int shift;    // the twiddle exponent's scale to the 2^m table: 2^shift
};

// x *= w_(2^(base + S))^(k' l), k' = register bits [0, base), l = bits
// [base, base + S) read from the top down
__global__ void __launch_bounds__(256) k_digit_twiddle(const __grid_constant__ TwArgs a) {
    const uint64_t hmask = (1ull << a.h) - 1ull;
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < a.count;
         i += (uint64_t)gridDim.x * blockDim.x) {
        const uint64_t r = i >> a.lo;
        const uint64_t kp = r & ((1ull << a.base) - 1ull);
        const uint64_t l = __brevll(r >> a.base) >> (64 - a.S);
        if (kp == 0 || l == 0) continue;
        // exponent over 2^(base + S): one table entry when the order is small
        // enough for a direct table, else the product of the two 2^m tables
        const uint64_t e0 = (kp * l) & ((1ull << (a.base + a.S)) - 1ull);
        double2 w;
        if (a.direct) {
            w = a.direct[e0];
        } else {
            const uint64_t e = e0 << a.shift;
            w = F64::cmul(a.coarse[e >> a.h], a.fine[e & hmask]);
        }
        a.x[i] = F64::cmul(w, a.x[i]);
    }
}

// Direct table of the 2^k roots of unity w_(2^k)^j (FP64-generated, stored in
// the policy's type), cached per (device, k, sign, policy) like the two-level
// tables; k <= 20 (16 MB for complex128, resident in L2).
template <class P>
__global__ void k_roots_direct(typename P::M* t, int k, int sign) {
    const uint64_t N = 1ull << k;
    for (uint64_t j = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; j < N; j += (uint64_t)gridDim.x * blockDim.x) {
        double sn, cs;
        sincospi(scalbn((double)j, 1 - k), &sn, &cs);
        t[j] = P::from_d(cs, sign > 0 ? sn : -sn);
    }
}
std::map<std::pair<int, TableKey>, void*> g_direct;   // (device, (k, sign, policy)) -> table

template <class P>
const typename P::M* get_direct(qe_state* s, int k, int sign, int pol) {
    int dev = 0;
    QE_CUDA(cudaGetDevice(&dev));
    auto key = std::make_pair(dev, TableKey{k, sign, pol});
    auto it = g_direct.find(key);
    if (it != g_direct.end()) return (const typename P::M*)it->second;
    void* t = nullptr;
    QE_CUDA(cudaMalloc(&t, sizeof(typename P::M) << k));
    Launch L(s, "fft_twiddles", 0.0, false);
    const unsigned grid = (unsigned)std::min<uint64_t>(((1ull << k) + 255) / 256, 4096);
    k_roots_direct<P><<<grid, 256, 0, s->stream>>>((typename P::M*)t, k, sign);
    QE_CUDA(cudaGetLastError());
    QE_CUDA(cudaStreamSynchronize(s->stream));   // once a table: later callers may be on other streams
    g_direct[key] = t;
    return (const typename P::M*)t;
}

}  // namespace

int qft_digits(int n, int m, int* digit, int* group) {
    const int G = (m + 4) / 5;
    // The lowest of five qubits, the others even (wider ones lowest: longer runs):
    // blocks are then filled up with register qubits only, and amplitudes that
    // differ outside a register of five qubits or more, however different in size,
    // share no scale.  (A lowest digit of three or four, with all of the
    // register above it choosing its matrix, took in qubits outside: a branch
    // 2^-30 of its neighbour kept 26 bits.)
    if (G > 1) digit[G - 1] = 5;
    for (int j = 0, r = G > 1 ? m - 5 : m, k = std::max(1, G - 1); j < k; ++j) digit[j] = r / k + (j >= k - r % k ? 1 : 0);
    auto fits = [&](int P, int d) { return P == 0 || (P <= n - 16 && P + d <= 20); };
    // the fewest groups, each as long as it can be ...
    int groups = 0;
    for (int j = 0; j < G; ++groups)
        for (int P = 0; j < G && fits(P, digit[j]); P += digit[j++]) group[j] = groups;
    // ... then as even as possible, where every digit still fits
    int even[7];
    bool ok = true;
    for (int g = 0, j = 0; g < groups; ++g)
        for (int P = 0; j < G * (g + 1) / groups; P += digit[j++]) {
            ok &= fits(P, digit[j]);
            even[j] = g;
        }
    if (ok) std::copy(even, even + G, group);
    return G;
}

namespace {

void qft_tc(qe_state* s, int lo, int m, int inverse) {
    const int sign = inverse ? -1 : 1;
    int digit[7], group[7];
    const int G = qft_digits(s->n, m, digit, group), groups = group[G - 1] + 1;
    static thread_local TwArgs a;
    a.x = reinterpret_cast<double2*>(s->d);
    a.count = dim(s);
    a.lo = lo;
    a.h = (m + 1) / 2;
    int top = m, j = 0;
    for (int g = 0; g < groups; ++g) {
        int P = 0;
        for (; j < G && group[j] == g; ++j) {
            const int d = digit[j];
            top -= d;
            launch_dft_digit_c128(s, lo, lo + top, d, P, G > 1, get_direct<F64>(s, P + d, sign, 1));
            P += d;
        }
        if (top == 0) break;
        a.base = top;
        a.S = P;
        a.shift = m - (top + P);
        a.direct = (top + P <= 20) ? get_direct<F64>(s, top + P, sign, 1) : nullptr;
        if (!a.direct) {
            const Table tb = get_tables<F64>(s, m, sign, 1);
            a.fine = (const double2*)tb.fine;
            a.coarse = (const double2*)tb.coarse;
        }
        const unsigned grid = (unsigned)std::min<uint64_t>((a.count + 255) / 256, (uint64_t)num_sms() * 8);
        Launch L(s, "fft_twiddle", 2.0 * dim(s) * amp_bytes(s));
        k_digit_twiddle<<<grid, 256, 0, s->stream>>>(a);
        QE_CUDA(cudaGetLastError());
    }
    if (G > 1) bitrev_impl<F64>(s, lo, m, "digitrev");
}

}  // namespace

// Digit passes on the tensor cores or the radix-2 shared-memory transform, for
// complex128 registers of at least 3 qubits on states of at least 12.  A digit
// pass takes about 15 us on a small state and 1/0.24 of the copy time on a large
// one; a shared-memory pass (11 stages, 8 to 10 above low qubits) costs the
// arithmetic of its stages.  Measured (ms, shared memory / digits):
//   FP64 mode, one shared-memory pass: n = 18, m = 11 0.041 / 0.088, n = 20
//   0.127 / 0.105, n = 24 1.52 / 0.63; n = 20, m = 5 0.06 / 0.038;
//   several passes: n = 17, m = 17 0.077 / 0.106, n = 19 0.141 / 0.120, n = 24,
//   m = 23 3.96 / 1.30 (registers of whole five-qubit digits above one pass
//   take the digits at every size);
//   double-float mode: n = 24, m = 5 0.294 / 0.195 (n = 20 0.031 / 0.038),
//   m = 10 0.439 / 0.483, m = 24 1.48 / 1.34, n = 20, m = 20 0.120 / 0.160,
//   n = 30, m = 30 118 / 79.
// Registers of three and four qubits share their blocks' scale with amplitudes
// outside the register; the double-float mode leaves them to the elementwise
// transform.
static bool qft_on_tensor_cores(const qe_state* s, int lo, int m) {
    if (s->dtype != QE_C128 || !s->c128_tc || !s->tensor_cores || s->force_tile || s->n < 12 || m < 3) return false;
    const bool one_pass = m <= 11 - std::min(lo, 3);
    if (s->arith == QE_ARITH_FP64) return one_pass ? s->n >= 20 : s->n >= 19 || m % 5 == 0;
    return m <= 5 ? m == 5 && s->n >= 22 : !one_pass && s->n >= 23;
}

void launch_qft_fft(qe_state* s, int lo, int m, int inverse) {
    const bool tc = qft_on_tensor_cores(s, lo, m);
    if (tc) {
        qft_tc(s, lo, m, inverse);
        return;
    }
    if (s->dtype == QE_C64 && m > kFft4Bits - std::min(lo, 3)) fft4(s, lo, m, inverse);
    else if (s->dtype == QE_C64) fft_impl<F32>(s, lo, m, inverse, 0);
    else if (s->arith == QE_ARITH_FP64) fft_impl<F64>(s, lo, m, inverse, 1);
    else fft_impl<DF>(s, lo, m, inverse, 2);
}

void launch_bitrev(qe_state* s, int lo, int m) {
    if (s->dtype == QE_C64) bitrev_impl<F32>(s, lo, m);
    else bitrev_impl<F64>(s, lo, m);   // pure data movement: storage type only
}

}  // namespace qe
