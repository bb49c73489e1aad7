// Expectation values of Pauli sums on large states (Sec. III-D): passes over
// the state by register sets of four qubits.
//
// A pass works on tiles of 2^12 amplitudes: two sets A and B of four qubits and
// the four lowest others, the row.  A thread first holds the 16 amplitudes that
// differ in A, as loaded (rows of 256 bytes, 128 complex64); they go to shared
// memory and come back as the 16 that differ in B, and in one pass as those
// that differ in the row (qubits 0 to 3).  Every term whose X/Y qubits lie in the
// set held pairs two of the thread's registers.  One pass also sums the Z-only
// terms.  Terms of one pattern (X X and Y Y) share their products.
//
// Three arithmetics, each with the precision of the path it stands in for:
//   complex128 sums whose terms all fit the register rounds: fixed point.  With E
//     the largest biased exponent of the tile's components, q = v 2^(1076 - E)
//     rounded to the nearest, |q| < 2^54, in the limbs q = h 2^28 + l.  The products
//     h h' at unit 2^56, h l' + l h' at unit 2^28 and l l' are summed exactly in 64
//     bits.  (Without l l' the sums of states that span many binary orders came out
//     2 to 4 10^-15 short, as in the register rounds; with it they are off by a few
//     10^-17.)  A weight's sum goes to FP64 once a tile: three instructions on the
//     FP64 pipe (two lanes a clock and SM) for 16 amplitudes a thread.  The four
//     single X of a set are eight products of an amplitude of even parity with the
//     sum of its four odd neighbours instead of 32 products.
//   other complex128 sums: FP64 products, two multiply-adds a pair (in fixed point
//     a term that pairs one large with one small amplitude of a tile would lose
//     the small one's digits).
//   complex64: exact products as pairs of floats, summed with their errors.
//
// Fixed point is bound by instruction issue at 16 warps an SM (registers), the
// ALU pipe first: about 100 instructions an amplitude and pass, 36 of them the
// limbs; FP64 products by their pipe (90 % busy); the pairs of floats (ten packed
// instructions a pair) by latency, the ALU pipe 46 and the FMA pipe 40 % busy at
// 16 warps an SM.  n = 28, against the other path
// (register rounds in fixed point, or tiles with FP64 or float-pair products):
// transverse-field Ising complex128 9.42 -> 4.31 ms, complex64 8.31 -> 4.7;
// Heisenberg chain with unequal couplings 33.3 -> 20.0 and 19.7 -> 6.4, with equal
// ones (X X + Y Y is then half the pairs) 32.2 -> 10.5 and 18.9 -> 4.0.  In fixed
// point the Heisenberg chain took 12.2 ms.  Sets of four qubits by warps alone,
// without the shared tile, took 7.0 ms for Ising: limbs made anew for every set.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <type_traits>
#include <unordered_map>
#include <unordered_set>
#include <vector>

#include "qe_arith.cuh"
#include "qe_f32x2.cuh"
#include "qe_internal.h"

namespace qe {

namespace {

constexpr int kTile = 12, kThreads = 256, kPerSm = 2;   // bits of a tile; threads; blocks an SM
constexpr int kTerms = 96, kMasks = 64, kGroups = 16;   // a pass: sums of pairs, Z masks, their weights
// states of at least 17 qubits: 32 tiles.  There Ising 0.062 ms a call against 0.065 by
// register rounds, Heisenberg 0.097 against 0.142 by tiles; with fewer tiles
// the launches decide and the other paths take as few
constexpr int kExpectSetsMin = 17;
constexpr size_t kHeld = kTerms * 3 / 8;   // terms of a pass: three make at most eight sums of pairs
constexpr int kMany = 256;       // terms of a list that is worth tables and a first estimate
constexpr uint32_t kZero = 64;   // biased FP64 exponent below which a tile's amplitudes count as zero

// Some pairs (j, j ^ xt) of the register set, all of one weight: the terms of a
// pattern and of the same Z bits outside the set share their products, each
// pair weighed by the sum of the terms' signed coefficients
struct Term {
    double w;             // > 0, twice the sum of the coefficients (its arithmetic's form); pairs of weight 0 are left out
    uint64_t zm;          // Z bits outside the set
    uint32_t sel : 16;    // the pairs, by the j without xt's lowest bit
    uint32_t xt : 4;      // X/Y bits in the set; 0: the sum of its four single X
    uint32_t im : 1, neg : 1, flip : 1, fold : 1;   // flip: neg or zm
};
// The Z masks of a weight whose bits in A are the same: n masks (bits of m). With
// k of them odd outside A at the thread's place, the amplitudes j of odd
// parity in A have n - k odd masks and the others k; pat holds the parities, a byte
// each
struct ZPattern {
    uint64_t m;
    uint32_t n, pat[4];
};
struct ZGroup {
    double w;             // the weight (its arithmetic's form; twice it in fixed point)
    int c0, c1, masks;    // patterns [c0, c1), at most 64 masks
};
template <class S>
struct Args {
    const S* x;
    uint8_t q[3][4];      // the qubits of A and B and the tile's four others ("row")
    int t[4];             // terms over A [t[0], t[1]), over B [t[1], t[2]), over the row [t[2], t[3])
    int nz, nzg;          // Z masks and weights
    int item_log2;        // tiles an item
    uint64_t items, places;   // places: the qubits outside the tile
    Term term[kTerms];
    ZGroup g[kGroups];
    ZPattern c[kMasks];
    uint64_t z[kMasks];
    double* partial;
};

__device__ __forceinline__ uint32_t top_bits(double2 v) {
    return max((uint32_t)__double2hiint(v.x) & 0x7FFFFFFFu, (uint32_t)__double2hiint(v.y) & 0x7FFFFFFFu);
}
// Limbs of a component d binary orders below the largest, its mantissa with the
// leading bit at bit 63 of (hi, lo): h the top 26 bits of the window, l the rest,
// rounded (2^28 not carried over).  The products with the sign (+1 or -1) run
// on the FMA pipe; the shifts and masks on the ALU pipe (64 lanes a clock) are
// what bounds a pass
__device__ __forceinline__ void limbs(uint32_t hi, uint32_t lo, uint32_t d, int sign, int& h, int& l) {
    const uint32_t x = (uint32_t)shift_down((((uint64_t)hi << 32) | lo), d + 9u) & 0x1FFFFFFFu;
    const int sg = sign | 1;
    h = (int)shift_down(hi, d + 6u) * sg;
    l = (int)((x + 1u) >> 1) * sg;
}
__device__ __forceinline__ void limbs_of(double v, uint32_t E, int& h, int& l) {
    const uint32_t hi = (uint32_t)__double2hiint(v), lo = (uint32_t)__double2loint(v);
    const uint32_t d = E - ((hi & 0x7FFFFFFFu) >> 20);
    limbs(__funnelshift_l(lo, (hi & 0xFFFFFu) | 0x100000u, 11), lo << 11, d, (int)hi >> 31, h, l);
}

__device__ __forceinline__ double pow2(int x) { return __hiloint2double(min(x, 2047) << 20, 0); }   // 2^(x - 1023), x >= 1

// Times in ms at n = 26: a pass; the Z masks of a weight (the other path: a mask);
// a term; eight of its pairs.
// launch: what a pass takes at any size
struct Cost {
    double pass, masks, term, pairs, launch;
};

// The three arithmetics: S an amplitude in memory, V one as held, Acc a sum of
// products, Sum a thread's sum of weighted Accs.  pair_add: a += Re (IM: Im) of
// conj(w) v; add: a += t or -= t.
struct Fixed {
    using S = double2;
    struct alignas(16) V {
        int xh, xl, yh, yl;
    };
    struct Acc {
        long long h0 = 0, h1 = 0, m0 = 0, m1 = 0, ll = 0;   // ll: one term's, then into m0
    };
    using Sum = double;
    static constexpr bool kFixed = true;
    static constexpr Cost kCost = {0.25, 0.06, 0.034, 0.0, 0.005}, kOther = {0.35, 0.01, 0.045, 0.0, 0.005};
    static double weight(double w) { return w; }
    template <bool IM>
    __device__ __forceinline__ static void pair_add(Acc& a, const V& w, const V& v) {
        if constexpr (!IM) {
            a.h0 += (long long)w.xh * v.xh;
            a.h1 += (long long)w.yh * v.yh;
            a.m0 += (long long)w.xh * v.xl;
            a.m0 += (long long)w.xl * v.xh;
            a.m1 += (long long)w.yh * v.yl;
            a.m1 += (long long)w.yl * v.yh;
            a.ll += (long long)w.xl * v.xl;
            a.ll += (long long)w.yl * v.yl;
        } else {
            a.h0 += (long long)w.xh * v.yh;
            a.h1 -= (long long)w.yh * v.xh;
            a.m0 += (long long)w.xh * v.yl;
            a.m0 += (long long)w.xl * v.yh;
            a.m1 -= (long long)w.yh * v.xl;
            a.m1 -= (long long)w.yl * v.xh;
            a.ll += (long long)w.xl * v.yl;
            a.ll -= (long long)w.yl * v.xl;
        }
    }
    __device__ __forceinline__ static void term_end(Acc& a) {
        a.m0 += a.ll >> 28;   // at most 2^62
        a.ll = 0;
    }
    __device__ __forceinline__ static void add(Acc& a, const Acc& t, uint32_t neg) {
        const long long f = -(long long)neg;
        a.h0 += (t.h0 ^ f) - f;
        a.h1 += (t.h1 ^ f) - f;
        a.m0 += (t.m0 ^ f) - f;
        a.m1 += (t.m1 ^ f) - f;
    }
    // s += z w 2^(2 E - 2096)
    __device__ __forceinline__ static void fold(Sum& s, long long z, double w, int E) {
        if (E > 800 && E < 1250) s = __fma_rn((double)z, __dmul_rn(w, pow2(2 * E - 1073)), s);
        else s = __fma_rn(__dmul_rn(__dmul_rn((double)z, pow2(E + 3)), w), pow2(E - 53), s);
    }
    __device__ __forceinline__ static void fold(Sum& s, const Acc& a, double w, int E) {
        fold(s, a.h0 + a.h1 + ((a.m0 + a.m1 + (1ll << 27)) >> 28), w, E);
    }
    __device__ __forceinline__ static double total(Sum s) { return s; }
};
struct Native {
    using S = double2;
    using V = double2;
    struct Acc {
        double a = 0.0, b = 0.0;
    };
    using Sum = double;
    static constexpr bool kFixed = false;
    static constexpr Cost kCost = {0.11, 0.5, 0.02, 0.1, 0.012}, kOther = {0.2, 0.015, 0.102, 0.0, 0.022},
                          kOtherDf = {0.35, 0.0095, 0.061, 0.0, 0.022};
    static double weight(double w) { return w; }
    __device__ __forceinline__ static V held(double2 v) { return v; }
    template <bool IM>
    __device__ __forceinline__ static void pair_add(Acc& a, const V& w, const V& v) {
        a.a = __fma_rn(w.x, IM ? v.y : v.x, a.a);
        a.b = __fma_rn(w.y, IM ? -v.x : v.y, a.b);
    }
    __device__ __forceinline__ static void term_end(Acc&) {}
    __device__ __forceinline__ static void add(Acc& a, const Acc& t, uint32_t neg) {
        const int sg = (int)(neg << 31);
        a.a += __hiloint2double(__double2hiint(t.a) ^ sg, __double2loint(t.a));
        a.b += __hiloint2double(__double2hiint(t.b) ^ sg, __double2loint(t.b));
    }
    // a += n |v|^2 (n as a double by an addition: the conversion instruction takes
    // as long as a dozen)
    __device__ __forceinline__ static void count_add(Acc& a, const V& v, int n) {
        const double c = __dadd_rn(__hiloint2double(0x43380000 + (n >> 31), n), -6755399441055744.0);   // 1.5 2^52
        a.a = __fma_rn(__fma_rn(v.x, v.x, __dmul_rn(v.y, v.y)), c, a.a);
    }
    __device__ __forceinline__ static void fold(Sum& s, const Acc& a, double w, int) { s = __fma_rn(a.a + a.b, w, s); }
    __device__ __forceinline__ static double total(Sum s) { return s; }
};
// Pairs of floats, a component a lane: products exact (product and residual),
// sums by TwoSum with the errors summed beside them
struct Pairs {
    using S = float2;
    using V = f2;
    struct Acc {
        f2 s = 0, e = 0;
    };
    using Sum = Acc;
    static constexpr bool kFixed = false;
    static constexpr Cost kCost = {0.19, 0.085, 0.011, 0.0065, 0.012}, kOther = {0.19, 0.0045, 0.04, 0.0, 0.022};
    static double weight(double w) {   // as a pair of floats in a double's bits
        const float h = (float)w, l = (float)(w - (double)h);
        double r;
        std::memcpy(&r, &h, 4);
        std::memcpy(reinterpret_cast<char*>(&r) + 4, &l, 4);
        return r;
    }
    __device__ __forceinline__ static V held(float2 v) { return pack2(v.x, v.y); }
    // a += -n + l
    __device__ __forceinline__ static void take(Acc& a, f2 n, f2 l) {
        const f2 s = sub2(a.s, n), bb = sub2(s, a.s);
        const f2 err = sub2(sub2(a.s, sub2(s, bb)), add2(n, bb));
        a.s = s;
        a.e = add2(a.e, add2(err, l));
    }
    template <bool IM>
    __device__ __forceinline__ static void pair_add(Acc& a, const V& w, const V& v) {
        f2 x = w, y = v;
        if constexpr (IM) {
            x ^= 0x8000000000000000ull;   // (w.x, -w.y)
            y = swap2(v);
        }
        const f2 n = mul2(neg2(x), y);
        take(a, n, fma2(x, y, n));
    }
    __device__ __forceinline__ static void term_end(Acc&) {}
    __device__ __forceinline__ static void add(Acc& a, const Acc& t, uint32_t neg) {
        const f2 m = neg ? 0ull : 0x8000000080000000ull;
        take(a, t.s ^ m, neg2(t.e ^ m));
    }
    __device__ __forceinline__ static void count_add(Acc& a, const V& v, int n) {
        const f2 f = dup2((float)n);
        const f2 h = mul2(v, v), l = fma2(v, v, neg2(h)), p = mul2(neg2(h), f);
        take(a, p, fma2(l, f, fma2(h, f, p)));
    }
    __device__ __forceinline__ static void fold(Sum& s, const Acc& a, double w, int) {
        const f2 wh = dup2(__int_as_float(__double2loint(w))), wl = dup2(__int_as_float(__double2hiint(w)));
        const f2 n = mul2(neg2(wh), a.s);
        take(s, n, fma2(wl, a.s, fma2(wh, a.e, fma2(wh, a.s, n))));
    }
    __device__ __forceinline__ static double total(Sum s) {
        const float2 a = unpack2(s.s), b = unpack2(s.e);
        return ((double)a.x + (double)b.x) + ((double)a.y + (double)b.y);
    }
};

// The pairs of a pattern fall in two halves by the parity of j's bits in it: X X
// and Y Y of different weights weigh them differently, of equal weights cancel in
// one.  A half that a term leaves out whole is jumped over (an FP64
// instruction that is only predicated off takes the pipe's time all the same).
template <int XT, bool ODD>
__host__ __device__ constexpr uint32_t half_of() {
    uint32_t m = 0;
    for (int j = 0; j < 16; ++j) {
        const int b = j & XT, odd = (b ^ (b >> 1) ^ (b >> 2) ^ (b >> 3)) & 1;
        if (!(j & (XT & -XT)) && (odd != 0) == ODD) m |= 1u << j;
    }
    return m;
}
template <class P, int XT, bool IM, uint32_t HALF>
__device__ __forceinline__ void half_pairs(const typename P::V (&v)[16], uint32_t sel, typename P::Acc& a) {
    if constexpr (HALF != 0) {
        if (sel & HALF) {
#pragma unroll
            for (int j = 0; j < 16; ++j)
                if (((HALF >> j) & 1u) && ((sel >> j) & 1u)) P::template pair_add<IM>(a, v[j ^ XT], v[j]);
        }
    }
}
template <class P, int XT, bool IM>
__device__ __forceinline__ void pairs(const typename P::V (&v)[16], uint32_t sel, typename P::Acc& a) {
    if constexpr (P::kFixed) {   // no slower for the few pairs that are predicated off
        half_pairs<P, XT, IM, half_of<XT, false>() | half_of<XT, true>()>(v, sel, a);
    } else {
        half_pairs<P, XT, IM, half_of<XT, false>()>(v, sel, a);
        half_pairs<P, XT, IM, half_of<XT, true>()>(v, sel, a);
    }
}
template <class P, int XT>
__device__ __forceinline__ void term(const typename P::V (&v)[16], uint32_t sel, bool im, typename P::Acc& a) {
    if (im) pairs<P, XT, true>(v, sel, a);
    else pairs<P, XT, false>(v, sel, a);
}
// the four single X of a set (fixed point, whose sums of four are exact)
__device__ __forceinline__ void chain(const Fixed::V (&v)[16], Fixed::Acc& a) {
#pragma unroll
    for (int j = 0; j < 16; ++j) {
        if (((j >> 3) ^ (j >> 2) ^ (j >> 1) ^ j) & 1) continue;
        const Fixed::V &b = v[j ^ 1], &c = v[j ^ 2], &d = v[j ^ 4], &e = v[j ^ 8];
        const Fixed::V w{(b.xh + c.xh) + (d.xh + e.xh), (b.xl + c.xl) + (d.xl + e.xl), (b.yh + c.yh) + (d.yh + e.yh),
                         (b.yl + c.yl) + (d.yl + e.yl)};
        Fixed::pair_add<false>(a, w, v[j]);
    }
}

// bits of v at the set bits of m, lowest first
__device__ __forceinline__ uint64_t deposit(uint64_t v, uint64_t m) {
    uint64_t x = 0;
    for (; m != 0 && v != 0; m &= m - 1, v >>= 1)
        if (v & 1ull) x |= m & (~m + 1ull);
    return x;
}

// Tile index bits: A (a lane's 16 registers), B (warp and top lane bit), row (low
// lane bits).  Held amplitudes lie at slot (A, B, row ^ B) of the shared tile, so
// that each of the three ways a thread's 16 amplitudes are read or written is
// free of bank conflicts (phases of 8 lanes of 16 bytes, 16 of 8).
template <class P>
__global__ void __launch_bounds__(kThreads, kPerSm) k_expect_sets(const __grid_constant__ Args<typename P::S> a) {
    using S = typename P::S;
    using V = typename P::V;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    constexpr uint32_t kSwz = sizeof(V) == 16 ? 7u : 15u;
    V* const tile = reinterpret_cast<V*>(smem_raw);
    __shared__ __align__(16) uint32_t s_top[kThreads / 32];
    __shared__ uint32_t s_odd[2];
    __shared__ double sh[kThreads / 32];
    const uint32_t tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5;
    const uint32_t lo4 = tid & 15u, hi4 = tid >> 4;
    typename P::Sum s{};
    auto spread = [&](uint32_t v, const uint8_t (&q)[4]) {
        uint64_t x = 0;
#pragma unroll
        for (int b = 0; b < 4; ++b) x |= (uint64_t)((v >> b) & 1u) << q[b];
        return x;
    };
    const uint64_t own = spread(hi4, a.q[1]) | spread(lo4, a.q[2]);   // of the tile's loads: B and row
    const uint64_t line = spread(hi4, a.q[0]) | spread(lo4, a.q[1]);  // of its prefetches: A and B
    uint64_t zown = 0;   // parities of the masks' bits in B and the row
    for (int m = 0; m < a.nz; ++m) zown |= (uint64_t)(__popcll(own & a.z[m]) & 1) << m;
    const uint64_t o0 = 1ull << a.q[0][0], o1 = 1ull << a.q[0][1], o2 = 1ull << a.q[0][2], o3 = 1ull << a.q[0][3];
    for (uint64_t item = blockIdx.x; item < a.items; item += gridDim.x) {
        uint64_t place = deposit(item << a.item_log2, a.places);
        for (int i = 0; i < (1 << a.item_log2); ++i) {
            const uint64_t base = own | place;
            S raw[16];
            {
                const S* const x0 = a.x + base;
#pragma unroll
                for (int j = 0; j < 16; ++j)
                    raw[j] = __ldg(x0 + ((j & 1 ? o0 : 0) + (j & 2 ? o1 : 0) + (j & 4 ? o2 : 0) + (j & 8 ? o3 : 0)));
            }
            const uint64_t here = place;
            place = ((place | ~a.places) + 1ull) & a.places;
            if (i + 1 < (1 << a.item_log2)) {
                const char* const nx = reinterpret_cast<const char*>(a.x + (line | place));
                asm volatile("prefetch.global.L2 [%0];" ::"l"(nx));
                if constexpr (sizeof(S) == 16) {
                    asm volatile("prefetch.global.L2 [%0];" ::"l"(nx + 128));
                }
            }
            uint32_t top = 0u;
            if constexpr (P::kFixed) {
#pragma unroll
                for (int j = 0; j < 16; ++j) top = max(top, top_bits(raw[j]));
                top = __reduce_max_sync(0xffffffffu, top);
                if (lane == 0) s_top[warp] = top;
            }
            if (a.nz > 0 && warp < 2) {   // parities of the masks at the tile's place
                const uint64_t m = warp * 32 + lane < (uint32_t)a.nz ? a.z[warp * 32 + lane] : 0ull;
                const uint32_t odd = __ballot_sync(0xffffffffu, __popcll(here & m) & 1);
                if (lane == 0) s_odd[warp] = odd;
            }
            __syncthreads();   // also: the previous tile has been read
            int E = 0;
            V v[16];
            if constexpr (P::kFixed) {
                const uint4 u = *reinterpret_cast<const uint4*>(&s_top[0]), w = *reinterpret_cast<const uint4*>(&s_top[4]);
                top = max(max(max(u.x, u.y), max(u.z, u.w)), max(max(w.x, w.y), max(w.z, w.w)));
                E = (int)(top >> 20);
                // the same for all threads: infinities, NaN; zero
                const bool bad = E == 0x7FF;
                if (bad) s = __hiloint2double(0x7FF80000, 0);
                if (bad || E < (int)kZero) {
                    __syncthreads();   // s_top is written again
                    continue;
                }
#pragma unroll
                for (int j = 0; j < 16; ++j) {
                    limbs_of(raw[j].x, (uint32_t)E, v[j].xh, v[j].xl);
                    limbs_of(raw[j].y, (uint32_t)E, v[j].yh, v[j].yl);
                }
            } else {
#pragma unroll
                for (int j = 0; j < 16; ++j) v[j] = P::held(raw[j]);
            }
            if (a.t[3] > a.t[1]) {
#pragma unroll
                for (int j = 0; j < 16; ++j)
                    tile[((uint32_t)j * 16u + hi4) * 16u + (lo4 ^ (hi4 & kSwz))] = v[j];
            }
            const uint64_t zbits = zown ^ ((uint64_t)s_odd[1] << 32 | s_odd[0]);
#pragma unroll 1
            for (int g = 0; g < a.nzg; ++g) {
                // odd masks of each amplitude, four counts a word
                uint32_t odd[4] = {0, 0, 0, 0}, even = 0;
                const int masks = a.g[g].masks;
#pragma unroll 1
                for (int c = a.g[g].c0; c < a.g[g].c1; ++c) {
                    const uint32_t k = (uint32_t)__popcll(zbits & a.c[c].m), up = a.c[c].n - 2u * k;
                    even += k;
#pragma unroll
                    for (int w = 0; w < 4; ++w) odd[w] += a.c[c].pat[w] * up;   // no byte leaves [0, 64] in the end
                }
#pragma unroll
                for (int w = 0; w < 4; ++w) odd[w] += even * 0x01010101u;
                if constexpr (P::kFixed) {
                    long long z[2] = {0, 0};   // each at most 2^62
#pragma unroll
                    for (int j = 0; j < 16; ++j) {
                        // |q|^2 at unit 2^56
                        const long long hh = (long long)v[j].xh * v[j].xh + (long long)v[j].yh * v[j].yh;
                        const long long hl = (long long)v[j].xh * v[j].xl + (long long)v[j].yh * v[j].yl;
                        const long long ll = (long long)v[j].xl * v[j].xl + (long long)v[j].yl * v[j].yl;
                        const long long q2 = hh + ((hl + (ll >> 29) + (1ll << 26)) >> 27);
                        const int cnt = masks - 2 * (int)((odd[j >> 2] >> (8 * (j & 3))) & 0xFFu);
                        z[j & 1] += (long long)cnt * q2;
                    }
                    // half the sum, to even: cut off, every thread's tile loses a quarter unit, 10^-16 at n = 24
                    long long half = (z[0] >> 1) + (z[1] >> 1) + (z[0] & z[1] & 1);
                    half += (z[0] ^ z[1]) & half & 1;
                    P::fold(s, half, a.g[g].w, E);
                } else {
                    typename P::Acc z;
#pragma unroll
                    for (int j = 0; j < 16; ++j)
                        P::count_add(z, v[j], masks - 2 * (int)((odd[j >> 2] >> (8 * (j & 3))) & 0xFFu));
                    P::fold(s, z, a.g[g].w, 0);
                }
            }
            __syncthreads();
            typename P::Acc acc;
#pragma unroll 1
            for (int round = 0; round < 3; ++round) {
                const int k0 = a.t[round], k1 = a.t[round + 1];
                if (k0 == k1) continue;
                uint64_t mine = base;
                if (round == 1) {          // registers: B; thread: (A, row)
                    mine = here | spread(hi4, a.q[0]) | spread(lo4, a.q[2]);
#pragma unroll
                    for (int j = 0; j < 16; ++j) v[j] = tile[(hi4 * 16u + (uint32_t)j) * 16u + (lo4 ^ ((uint32_t)j & kSwz))];
                } else if (round == 2) {   // registers: the row; thread: (A, B)
                    mine = here | spread(hi4, a.q[0]) | spread(lo4, a.q[1]);
#pragma unroll
                    for (int j = 0; j < 16; ++j) v[j] = tile[tid * 16u + ((uint32_t)j ^ (lo4 & kSwz))];
                }
#pragma unroll 1
                for (int k = k0; k < k1; ++k) {
                    const Term& t = a.term[k];
                    const typename P::Acc old = acc;
                    const bool flip = t.flip;
                    if (flip) acc = typename P::Acc{};
                    const uint32_t sel = t.sel;
                    const bool im = t.im;
                    switch (t.xt) {
                        case 0:
                            if constexpr (P::kFixed) chain(v, acc);
                            break;
                        case 1: term<P, 1>(v, sel, im, acc); break;
                        case 2: term<P, 2>(v, sel, im, acc); break;
                        case 3: term<P, 3>(v, sel, im, acc); break;
                        case 4: term<P, 4>(v, sel, im, acc); break;
                        case 5: term<P, 5>(v, sel, im, acc); break;
                        case 6: term<P, 6>(v, sel, im, acc); break;
                        case 7: term<P, 7>(v, sel, im, acc); break;
                        case 8: term<P, 8>(v, sel, im, acc); break;
                        case 9: term<P, 9>(v, sel, im, acc); break;
                        case 10: term<P, 10>(v, sel, im, acc); break;
                        case 11: term<P, 11>(v, sel, im, acc); break;
                        case 12: term<P, 12>(v, sel, im, acc); break;
                        case 13: term<P, 13>(v, sel, im, acc); break;
                        case 14: term<P, 14>(v, sel, im, acc); break;
                        default: term<P, 15>(v, sel, im, acc); break;
                    }
                    P::term_end(acc);
                    if (flip) {
                        const typename P::Acc one = acc;
                        acc = old;
                        P::add(acc, one, (uint32_t)(__popcll(mine & t.zm) & 1) ^ t.neg);
                    }
                    if (t.fold) {
                        P::fold(s, acc, t.w, E);
                        acc = typename P::Acc{};
                    }
                }
            }
        }
    }
    double d = P::total(s);
    for (int o = 16; o > 0; o >>= 1) d += __shfl_down_sync(0xffffffffu, d, o);
    if (lane == 0) sh[warp] = d;
    __syncthreads();
    if (tid == 0) {
        double r = 0.0;
        for (int w = 0; w < kThreads / 32; ++w) r += sh[w];
        a.partial[blockIdx.x] = r;
    }
}

// One block: Neumaier sums of the partials, thread t taking t, t + 256, ..., then
// a fixed tree.
__global__ void __launch_bounds__(256) k_sum(const double* __restrict__ partial, int count, double* __restrict__ out) {
    __shared__ double ss[256], cs[256];
    auto add = [](double& s, double& c, double x) {
        const double t = s + x;
        c += fabs(s) >= fabs(x) ? (s - t) + x : (x - t) + s;
        s = t;
    };
    double s = 0.0, c = 0.0;
    for (int i = threadIdx.x; i < count; i += 256) add(s, c, partial[i]);
    ss[threadIdx.x] = s;
    cs[threadIdx.x] = c;
    __syncthreads();
    for (int h = 128; h > 0; h >>= 1) {
        if ((int)threadIdx.x < h) {
            add(ss[threadIdx.x], cs[threadIdx.x], ss[threadIdx.x + h]);
            cs[threadIdx.x] += cs[threadIdx.x + h];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) out[0] = ss[0] + cs[0];
}

// ------------------------------------------------------------------- plan
struct Set {
    uint64_t q = 0;                    // four qubits
    std::vector<int> terms;
};
struct PassPlan {
    uint64_t q[2] = {0, 0};            // A, B
    std::vector<int> terms[3];         // over A, B, qubits 0 to 3
};
// Z masks of a weight, at most 64
struct ZPlan {
    double w;
    std::vector<uint64_t> masks;
};

void plan_z(int nterms, const uint64_t* xm, const uint64_t* zm, const double* cf, std::vector<ZPlan>& out) {
    std::unordered_map<double, size_t> open;   // a weight's last group
    for (int t = 0; t < nterms; ++t) {
        if (xm[t] != 0) continue;
        const auto [at, fresh] = open.emplace(cf[t], out.size());
        if (fresh || out[at->second].masks.size() == kMasks) {
            at->second = out.size();
            out.push_back(ZPlan{cf[t], {}});
        }
        out[at->second].masks.push_back(zm[t]);
    }
}

// `m` filled up to four qubits with the lowest ones from 4 on outside `not_in`.
uint64_t filled(int n, uint64_t m, uint64_t not_in) {
    for (int q = 4; q < n && __builtin_popcountll(m) < 4; ++q)
        if (!((not_in >> q) & 1ull)) m |= 1ull << q;
    return m;
}

// Passes of two disjoint register sets for the X/Y terms; false if a term has
// more than four X/Y qubits.
bool plan_sets(int n, int nterms, const uint64_t* xm, std::vector<PassPlan>& out) {
    std::vector<Set> sets;
    std::vector<int> row, order;
    for (int t = 0; t < nterms; ++t) {
        if (xm[t] == 0) continue;
        if (__builtin_popcountll(xm[t]) > 4) return false;
        if (xm[t] < 16) row.push_back(t);
        else order.push_back(t);
    }
    std::stable_sort(order.begin(), order.end(), [&](int x, int y) {
        return std::make_pair(__builtin_ctzll(xm[x]), xm[x]) < std::make_pair(__builtin_ctzll(xm[y]), xm[y]);
    });
    // each term to the first set that contains it, else to the first with room;
    // in long lists the first set of every subset is kept (of no fewer qubits
    // than the terms have), and which sets have room
    std::unordered_map<uint64_t, int> first;
    std::vector<int> room;
    int fewest = 4;
    for (int t : order) fewest = std::min(fewest, __builtin_popcountll(xm[t]));
    const bool many = (int)order.size() > kMany;
    if (many) first.reserve(order.size());
    for (int t : order) {
        int i = -1;
        if (many) {
            const auto at = first.find(xm[t]);
            if (at != first.end()) i = at->second;
        } else {
            for (size_t k = 0; k < sets.size() && i < 0; ++k)
                if ((sets[k].q & xm[t]) == xm[t]) i = (int)k;
        }
        if (i < 0) {
            for (size_t r = 0; r < room.size() && i < 0; ++r)
                if (__builtin_popcountll(sets[room[r]].q | xm[t]) <= 4) i = room[r];
            if (i < 0) {
                i = (int)sets.size();
                sets.push_back(Set{});
                room.push_back(i);
            }
            const uint64_t q = sets[i].q |= xm[t];
            if (__builtin_popcountll(q) == 4) room.erase(std::find(room.begin(), room.end(), i));
            for (uint64_t m = q; many && m != 0; m = (m - 1) & q) {
                if (__builtin_popcountll(m) < fewest) continue;
                int& f = first.emplace(m, i).first->second;
                f = std::min(f, i);
            }
        }
        sets[i].terms.push_back(t);
    }
    std::vector<bool> done(sets.size(), false);
    bool hosted = row.empty();
    for (size_t i = 0; i < sets.size(); ++i) {
        if (done[i]) continue;
        PassPlan p;
        // a set beside it: the next one without its qubits, not looked for too long
        size_t k = i + 1;
        for (int tries = 0; k < sets.size() && (done[k] || (sets[k].q & sets[i].q)); ++k)
            if (!done[k] && ++tries == 64) {
                k = sets.size();
                break;
            }
        for (size_t b = sets.size(); k >= sets.size() && sets.size() > i + 64 && b > std::max(sets.size() - 64, i + 1); --b)
            if (!done[b - 1] && !(sets[b - 1].q & sets[i].q)) k = b - 1;
        p.q[0] = filled(n, sets[i].q, k < sets.size() ? sets[k].q : 0ull);
        p.terms[0] = sets[i].terms;
        if (k < sets.size()) {
            done[k] = true;
            p.q[1] = sets[k].q;
            p.terms[1] = sets[k].terms;
        }
        p.q[1] = filled(n, p.q[1], p.q[0]);
        if (!hosted && !((p.q[0] | p.q[1]) & 15ull)) {
            hosted = true;
            p.terms[2] = row;
        }
        out.push_back(p);
    }
    if (!hosted || out.empty()) {   // qubits 0 to 3 (or nothing but Z terms) by themselves
        PassPlan p;
        p.q[0] = filled(n, 0ull, 0ull);
        p.q[1] = filled(n, 0ull, p.q[0]);
        p.terms[2] = hosted ? std::vector<int>{} : row;
        out.push_back(p);
    }
    return true;
}

template <class P>
class Launcher {
    using S = typename P::S;

public:
    Launcher(qe_state* s, const uint64_t* xm, const uint64_t* zm, const double* cf)
        : s_(s), xm_(xm), zm_(zm), cf_(cf) {}

    // a power of two taken out of the weights (pairs of floats have a float's range)
    int scale = 0;
    // the weights' least and largest magnitude
    double least = HUGE_VAL, most = 0.0;

    // launches: the passes, cut to the terms and masks of one
    void build(const std::vector<PassPlan>& plan, const std::vector<ZPlan>& z) {
        size_t zi = 0;
        for (size_t i = 0; i < plan.size() || zi < z.size(); ++i) {
            PassPlan p = i < plan.size() ? plan[i] : PassPlan{{plan[0].q[0], plan[0].q[1]}, {}};
            size_t at[3] = {0, 0, 0};
            bool more;
            do {
                PassPlan part{{p.q[0], p.q[1]}, {}};
                size_t held = 0;
                more = false;
                for (int r = 0; r < 3; ++r) {
                    for (; at[r] < p.terms[r].size() && held < kHeld; ++at[r], ++held)
                        part.terms[r].push_back(p.terms[r][at[r]]);
                    more |= at[r] < p.terms[r].size();
                }
                Args<S> g;
                fill(g, part);
                g.nz = g.nzg = 0;
                int nc = 0;
                for (; zi < z.size() && g.nzg < kGroups && g.nz + z[zi].masks.size() <= kMasks; ++zi) {
                    ZGroup& zg = g.g[g.nzg++];
                    zg.w = weight((P::kFixed ? 2.0 : 1.0) * z[zi].w);
                    zg.masks = (int)z[zi].masks.size();
                    zg.c0 = nc;
                    int at[16];
                    std::fill(at, at + 16, -1);
                    for (uint64_t m : z[zi].masks) {
                        const uint32_t in = gather(m, g.q[0]);
                        if (at[in] < 0) {
                            ZPattern& c = g.c[at[in] = nc++];
                            c = ZPattern{};
                            for (uint32_t j = 0; j < 16; ++j)
                                c.pat[j >> 2] |= (uint32_t)(__builtin_popcount(j & in) & 1) << (8 * (j & 3));
                        }
                        g.c[at[in]].m |= 1ull << g.nz;
                        ++g.c[at[in]].n;
                        for (int b = 0; b < 4; ++b) m &= ~(1ull << g.q[0][b]);
                        g.z[g.nz++] = m;
                    }
                    zg.c1 = nc;
                }
                launches.push_back(g);
            } while (more);
        }
    }

    double cost(double unit) const {   // unit: launch times at n = 26 are those of n times this
        double c = 0.0;
        for (const auto& g : launches) {
            c += P::kCost.pass + unit * P::kCost.launch + P::kCost.masks * g.nzg;
            for (int k = 0; k < g.t[3]; ++k) {
                const Term& t = g.term[k];
                int even = 0, odd = 0;   // pairs of the halves: half a term's cost each
                for (uint32_t j = 0; j < 16; ++j)
                    if ((t.sel >> j) & 1u) (__builtin_popcount(j & t.xt) & 1 ? odd : even) = 1;
                const double parts = __builtin_popcount(t.xt) > 1 ? 0.5 * (even + odd) : 1.0;
                c += t.xt == 0 ? 0.06 : P::kCost.term + P::kCost.pairs * parts;
            }
        }
        return c;
    }

    double run() {
        const size_t smem = sizeof(typename P::V) << kTile;
        QE_CUDA(cudaFuncSetAttribute(k_expect_sets<P>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        const unsigned most = (unsigned)(num_sms() * kPerSm);
        const unsigned grid = (unsigned)std::min<uint64_t>(most, launches[0].items);
        const size_t total = (size_t)grid * launches.size();
        double* const scr = (double*)ensure_scratch(s_, (total + 1) * sizeof(double));
        for (size_t i = 0; i < launches.size(); ++i) {
            launches[i].partial = scr + 1 + i * grid;
            Launch L(s_, sizeof(S) == 16 ? "expect_fx" : "expect_rounds", (double)dim(s_) * amp_bytes(s_));
            k_expect_sets<P><<<grid, kThreads, smem, s_->stream>>>(launches[i]);
            QE_CUDA(cudaGetLastError());
        }
        {
            Launch L(s_, "sum_partials", 0.0, false);
            k_sum<<<1, 256, 0, s_->stream>>>(scr + 1, (int)total, scr);
            QE_CUDA(cudaGetLastError());
        }
        double e = 0.0;
        QE_CUDA(cudaMemcpyAsync(&e, scr, sizeof(double), cudaMemcpyDeviceToHost, s_->stream));
        QE_CUDA(cudaStreamSynchronize(s_->stream));
        return std::ldexp(e, scale);
    }

private:
    qe_state* s_;
    const uint64_t *xm_, *zm_;
    const double* cf_;
    std::vector<Args<S>> launches;

    double weight(double w) {
        if (w != 0.0) {
            least = std::min(least, std::fabs(w));
            most = std::max(most, std::fabs(w));
        }
        return P::weight(std::ldexp(w, -scale));
    }
    static uint32_t gather(uint64_t m, const uint8_t (&q)[4]) {
        uint32_t r = 0;
        for (int b = 0; b < 4; ++b) r |= (uint32_t)((m >> q[b]) & 1ull) << b;
        return r;
    }
    // terms over the qubits q, by weight (in turn upwards and downwards, so that
    // a weight's sum goes on over two rounds); the four single X of a weight as one
    void add_terms(Args<S>& g, int& k, int& units, const std::vector<int>& ts, const uint8_t (&q)[4], bool down) {
        std::vector<Term> put;
        std::vector<int> single[4], rest;
        for (int t : ts) {
            const uint32_t x = gather(xm_[t], q);
            if (P::kFixed && zm_[t] == 0 && !(x & (x - 1u))) single[__builtin_ctz(x)].push_back(t);
            else rest.push_back(t);
        }
        for (size_t i = 0; i < single[0].size();) {
            const double w = cf_[single[0][i]];
            size_t at[4];
            bool all = true;
            for (int b = 0; b < 4; ++b) {
                at[b] = 0;
                while (at[b] < single[b].size() && cf_[single[b][at[b]]] != w) ++at[b];
                all &= at[b] < single[b].size();
            }
            if (!all) {
                ++i;
                continue;
            }
            for (int b = 0; b < 4; ++b) single[b].erase(single[b].begin() + at[b]);
            i = 0;
            Term r{};
            r.w = 2.0 * std::fabs(w);
            r.neg = w < 0;
            put.push_back(r);
        }
        for (auto& v : single) rest.insert(rest.end(), v.begin(), v.end());
        struct Unit {
            uint32_t xt, im;
            uint64_t zm;
            double w[16];
        };
        std::vector<Unit> us;
        for (int t : rest) {
            const uint32_t zl = gather(zm_[t], q);
            const int ny = __builtin_popcountll(xm_[t] & zm_[t]) & 3;
            Unit u{gather(xm_[t], q), (uint32_t)(ny & 1), zm_[t], {}};
            for (int b = 0; b < 4; ++b) u.zm &= ~(1ull << q[b]);
            size_t i = 0;
            while (i < us.size() && !(us[i].xt == u.xt && us[i].im == u.im && us[i].zm == u.zm)) ++i;
            if (i == us.size()) us.push_back(u);
            const double w = (ny == 1 || ny == 2) ? -2.0 * cf_[t] : 2.0 * cf_[t];
            for (uint32_t j = 0; j < 16; ++j) us[i].w[j] += (__builtin_popcount(j & zl) & 1) ? -w : w;
        }
        for (const Unit& u : us) {
            const size_t first = put.size();
            for (uint32_t j = 0; j < 16; ++j) {
                if ((j & (u.xt & (0u - u.xt))) || u.w[j] == 0.0) continue;
                const uint32_t neg = u.w[j] < 0.0;
                size_t i = first;
                while (i < put.size() && !(put[i].w == std::fabs(u.w[j]) && put[i].neg == neg)) ++i;
                if (i == put.size()) {
                    Term r{};
                    r.w = std::fabs(u.w[j]);
                    r.zm = u.zm;
                    r.xt = u.xt;
                    r.im = u.im;
                    r.neg = neg;
                    put.push_back(r);
                }
                put[i].sel |= 1u << j;
            }
        }
        std::stable_sort(put.begin(), put.end(), [&](const Term& x, const Term& y) { return down ? x.w > y.w : x.w < y.w; });
        for (Term& t : put) {
            t.flip = t.neg || t.zm != 0;
            // in fixed point a fold's sums stay below 2^62: eight terms of eight pairs
            const int u = t.xt == 0 ? 4 : 1;
            if (k > 0 && ((P::kFixed && units + u > 8) || g.term[k - 1].w != t.w)) {
                g.term[k - 1].fold = 1;
                units = 0;
            }
            units += u;
            g.term[k++] = t;
        }
    }
    void fill(Args<S>& g, const PassPlan& p) {
        const int n = s_->n;
        g.x = reinterpret_cast<const S*>(s_->d);
        uint64_t used = p.q[0] | p.q[1];
        for (int r = 0; r < 2; ++r)
            for (int q = 0, b = 0; q < n; ++q)
                if ((p.q[r] >> q) & 1ull) g.q[r][b++] = (uint8_t)q;
        for (int q = 0, b = 0; b < 4; ++q)
            if (!((used >> q) & 1ull)) {
                g.q[2][b++] = (uint8_t)q;
                used |= 1ull << q;
            }
        g.places = ((1ull << n) - 1ull) & ~used;
        // tiles an item: eight, fewer while that leaves blocks idle
        const uint64_t tiles = 1ull << (n - kTile), blocks = (uint64_t)num_sms() * kPerSm;
        g.item_log2 = 0;
        while (g.item_log2 < 3 && (tiles >> (g.item_log2 + 1)) >= 8 * blocks) ++g.item_log2;
        g.items = tiles >> g.item_log2;
        int k = 0, units = 0;
        for (int r = 0; r < 3; ++r) {
            g.t[r] = k;
            add_terms(g, k, units, p.terms[r], g.q[r], r & 1);
        }
        g.t[3] = k;
        if (k > 0) g.term[k - 1].fold = 1;
        for (int i = 0; i < k; ++i) g.term[i].w = weight(g.term[i].w);
    }
};

// Cost of a plan's passes and of its different strings, each by itself: one term,
// or two where Z bits in its set give its pairs both signs (each with half of the
// pairs, of one parity or of both).
template <class P>
double rough_cost(const std::vector<PassPlan>& plan, const uint64_t* xm, const uint64_t* zm, double unit) {
    struct Key {
        uint64_t x, z;
        bool operator==(const Key& k) const { return x == k.x && z == k.z; }
    };
    struct Hash {
        size_t operator()(const Key& k) const { return (k.x * 0x9E3779B97F4A7C15ull ^ k.z) * 0xD6E8FEB86659FD93ull >> 16; }
    };
    std::unordered_set<Key, Hash> seen;
    size_t count = 0, launches = 0;
    for (const PassPlan& p : plan) {
        size_t held = 0;
        for (const auto& ts : p.terms) held += ts.size();
        count += held;
        launches += std::max<size_t>(1, (held + kHeld - 1) / kHeld);
    }
    seen.reserve(count);
    double c = launches * (P::kCost.pass + unit * P::kCost.launch);
    for (const PassPlan& p : plan)
        for (int r = 0; r < 3; ++r) {
            const uint64_t q = r == 0 ? p.q[0] : r == 1 ? p.q[1] : 15ull;
            for (int t : p.terms[r]) {
                if (!seen.insert(Key{xm[t], (zm[t] & ~q) << 1 | (__builtin_popcountll(xm[t] & zm[t]) & 1)}).second) continue;
                const uint64_t low = xm[t] & (0ull - xm[t]), signs = zm[t] & q & ~low;
                if (P::kFixed && zm[t] == 0 && xm[t] == low) c += 0.015;   // a quarter of a chain
                else if (signs == 0) c += P::kCost.term + P::kCost.pairs;
                else c += 2 * P::kCost.term + (signs == (xm[t] & ~low) ? 1 : 2) * P::kCost.pairs;
            }
        }
    return c;
}

template <class P>
bool expect_impl(qe_state* s, int nterms, const uint64_t* xm, const uint64_t* zm, const double* cf, size_t other,
                 double* out) {
    std::vector<PassPlan> plan;
    if (!plan_sets(s->n, nterms, xm, plan)) return false;
    std::vector<ZPlan> z;
    plan_z(nterms, xm, zm, cf, z);
    const double unit = std::ldexp(1.0, 26 - s->n);
    Cost o = P::kOther;
    if constexpr (std::is_same_v<P, Native>)
        if (!c128_f64(s)) o = P::kOtherDf;
    int nx = 0;
    for (int t = 0; t < nterms; ++t) nx += xm[t] != 0;
    const double old = other * (o.pass + unit * o.launch) + nx * o.term + (nterms - nx) * o.masks;
    // nothing is built for long sums that the passes and the different strings alone
    // make too dear (10,000 random strings of four qubits at n = 20: 70 ms a call
    // with all launches built, 53 so, 48 of them the other path's launches)
    if (nterms > kMany && rough_cost<P>(plan, xm, zm, unit) > old) return false;
    Launcher<P> l(s, xm, zm, cf);
    if (sizeof(typename P::S) == 8) {
        double top = 0.0;
        for (int t = 0; t < nterms; ++t) top = std::max(top, std::fabs(cf[t]));
        if (top > 0.0) l.scale = std::ilogb(top);
    }
    l.build(plan, z);
    if (sizeof(typename P::S) == 8 && l.least < std::ldexp(l.most, -40)) return false;   // weights beyond a float's range
    if (l.cost(unit) > old) return false;
    *out = l.run();
    return true;
}

}  // namespace

bool expect_sets(qe_state* s, int nterms, const uint64_t* xm, const uint64_t* zm, const double* cf, size_t other,
                 bool fixed, double* out) {
    if (s->n < kExpectSetsMin) return false;
    if (s->dtype == QE_C64) return expect_impl<Pairs>(s, nterms, xm, zm, cf, other, out);
    if (fixed) return expect_impl<Fixed>(s, nterms, xm, zm, cf, other, out);
    return expect_impl<Native>(s, nterms, xm, zm, cf, other, out);
}

}  // namespace qe
