// Batch of parameterised circuits in one persistent launch (CUDA graph).
//
// Each circuit is the hardware-efficient ansatz: `layers` times (RY(theta),
// RZ(phi) on every qubit, then CZ on (q, q+1) for q = 0..n-2), started from
// |0...0>, and returns the energy of the transverse-field Ising Hamiltonian
// sum_i Z_i Z_{i+1} + h sum_i X_i (open chain), the expectation evaluated
// directly (Sec. III-D).
//
// Arithmetic of a layer.  Every RZ and CZ is diagonal, so a layer is n real
// rotations followed by one diagonal.
//   - A rotation is applied without its scale: with a, b the two amplitudes,
//       p = a + kappa b,  q = b - kappa a,
//     kappa = -tan(theta/2) when |tan| <= 1, leaving (p, q) = (out0, out1) / c;
//     else kappa = cot(theta/2), leaving (p, q) = (out1, -out0) / s: the two
//     outputs trade places, which is kept as a flip bit of that qubit ("slot
//     bit = logical bit ^ flip") instead of being moved.  |kappa| <= 1, and
//     two real multiply-adds an amplitude and gate replace the eight of the
//     complex 2 x 2 matrix RZ RY.
//   - The scales of all rotations (and the deviation of the rounded RZ phases
//     from modulus one, the same for both slot bits) are one number of the
//     circuit: the host keeps the squared norm of the unscaled state as a pair
//     of FP64 numbers and the energy is divided by it; only its power of two
//     is taken out of the amplitudes, exactly, layer by layer.  Scales folded
//     into rounded factors put the energies off by 2e-14 (double-float) and
//     3e-15 (FP64) relative; 0.5 to 1.5e-14 and 1.5e-15 without.
//   - The diagonal of the layer is the product over the qubits of a factor for
//     each slot bit (the sign of the flip and the RZ phase) times
//     (-1)^popcount(x & x >> 1) for logical x.  Two tables of at most 64 and
//     128 partial products (and one scalar for the bits outside a tile) give
//     an amplitude's factor with one complex product.
//   - Layer 0 acts on |0...0>, so its result is a product state: the same
//     tables with the factors (1, -kappa) folded in write it directly.
// Double-float values keep (re, im) of the high and of the low words in packed
// pairs, so that one f32x2 instruction serves both components.
// 512 circuits of 10..22 qubits, 8 layers: complex128 double-float 252 ms with
// the complex matrices, 74 ms so; FP64 1030 and 215 ms (its pipe's rate);
// complex64 66 and 25 ms.
//
// Work decomposition (one work queue, claimed in order with an atomic head):
//   - circuits of at most seven or eight qubits take a warp each, in a launch beside
//     (k_batch_tiny);
//   - a circuit with n <= T qubits is one item: its whole state lives in one
//     CTA's shared memory, HBM is never touched;
//   - a circuit with n > T qubits keeps its state in HBM and is processed in
//     2*(layers-1) + 1 passes over tiles of 2^T amplitudes: per layer from
//     layer 1 on a "low" pass (contiguous tiles, rotations of qubits < T) and
//     a "high" pass (tiles of 2^(2T-n)-amplitude chunks, rotations of qubits
//     >= T, then the diagonal); the first pass starts from the product state
//     instead of reading; the last high pass also accumulates the ZZ terms and
//     the X terms of the high qubits; a final read-only low pass adds the X
//     terms of the low qubits (layers = 1: one high pass writes the product
//     state).  The states are internal, so double-float pairs are stored as
//     they are.  Each pass is split into items of a few tiles.
//   - rotations are done a few at a time in registers: a thread owns the 2^G
//     amplitudes that differ in G bits.  The first such group of a pass reads
//     global memory and the last one writes it, so a pass makes one
//     shared-memory round trip fewer than it has groups.
// An item may start only when every item of the circuit's earlier passes has
// finished: CTAs wait on a per-circuit completion counter.  Large circuits
// are queued in waves of at most 64 or 256 MiB of state, pass-major inside a wave, with the small circuits spread between the
// passes; the dependencies of any claimed item were claimed earlier by
// running CTAs; waits are bounded and report a timeout.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <type_traits>
#include <vector>

#include "qe_batch.h"
#include "qe_f32x2.cuh"
#include "qe_internal.h"

namespace qe {

namespace {

struct Item {
    int circuit;
    uint32_t tile0, tile1;
    uint32_t dep;      // completed items of this circuit required before starting
    int slot;          // energy partial slot (or -1)
    uint32_t kind : 2;    // 0 small, 1 low layer pass, 2 high layer pass, 3 energy low pass
    uint32_t first : 1;   // the circuit's first pass (starts from the product state)
    uint32_t last : 1;    // its last high pass (energy)
    uint32_t layer : 28;
};

struct Circ {
    int n;
    int nitems;        // items of this circuit
    int slot0, nslots; // energy partial slots
    uint64_t state_off; // amplitude offset of its HBM state (large circuits)
    uint64_t u_off;     // offset of its rotations (layers * n entries)
    uint64_t f_off;     // offset of its flip masks (layers entries)
    double scale2;      // its energy / the energy of the kept amplitudes
};

// Each policy: V one amplitude (also its memory form), K a rotation's kappa,
// R kappa expanded for the device, rot the unscaled rotation, norm the
// renormalisation after a group of rotations, cmul, neg, and the energy sums.
struct BF32 {
    using V = f2;
    using K = float;
    using F = V;                             // a diagonal's factor
    static F make_f(double re, double im) { return make_v(re, im); }
    static double kept(double x) { return (double)(float)x; }
    __device__ __forceinline__ static F fmul(const F& a, const F& b) { return cmul(a, b); }
    __device__ __forceinline__ static V to_v(const F& f) { return f; }
    static constexpr int kGroup = 4;         // bits per register group
    static constexpr int kTiny = 8;          // qubits of a circuit that one warp takes
    static constexpr int kSw = 4;            // swizzle: 16 8-byte slots a row
    struct R { f2 k, nk; };
    static K make_k(double k) { return (float)k; }
    static double value(K k) { return (double)k; }
    static V make_v(double re, double im) {
        const float2 v = make_float2((float)re, (float)im);
        V r;
        std::memcpy(&r, &v, 8);
        return r;
    }
    __device__ __forceinline__ static R expand(K k) { return R{dup2(k), dup2(-k)}; }
    __device__ __forceinline__ static F one() { return pack2(1.f, 0.f); }
    __device__ __forceinline__ static void rot(V& a, V& b, const R& r) {
        const V p = fma2(r.k, b, a);
        b = fma2(r.nk, a, b);
        a = p;
    }
    // v + k u
    __device__ __forceinline__ static V step(const V& v, K k, uint32_t minus, const V& u) {
        return fma2(dup2(minus ? -k : k), u, v);
    }
    __device__ __forceinline__ static void norm(V&) {}
    __device__ __forceinline__ static V cmul(const V& w, const V& v) {
        const float2 f = unpack2(w);
        return fma2(dup2(f.x), v, mul2(pack2(-f.y, f.y), swap2(v)));
    }
    __device__ __forceinline__ static V neg(const V& v, uint32_t odd) {
        const uint32_t s = odd << 31;
        return v ^ (((f2)s << 32) | s);
    }
    __device__ __forceinline__ static void ld(V& v, const V* p) { v = __ldcg(p); }
};

// double-float pairs h + l, unnormalised: |l| a few units of h's last place
struct BDF {
    struct alignas(16) V { f2 h, l; };
    using K = float2;                        // (high, low)
    // The diagonal's factors, few and shared by many amplitudes, are multiplied
    // in FP64 (idle otherwise) and split once: a pair product's error of about
    // 2^-47 in a table entry would not average out over the amplitudes.
    using F = double2;
    static F make_f(double re, double im) { return make_double2(re, im); }
    static double kept(double x) { return x; }
    __device__ __forceinline__ static F fmul(const F& a, const F& b) {
        return make_double2(__fma_rn(a.x, b.x, -__dmul_rn(a.y, b.y)), __fma_rn(a.x, b.y, __dmul_rn(a.y, b.x)));
    }
    __device__ __forceinline__ static V to_v(const F& f) {
        const float x = (float)f.x, y = (float)f.y;
        return V{pack2(x, y), pack2((float)__dsub_rn(f.x, (double)x), (float)__dsub_rn(f.y, (double)y))};
    }
    static constexpr int kGroup = 3;
    static constexpr int kTiny = 7;
    static constexpr int kSw = 3;            // 8 16-byte slots a row
    struct R { f2 h, l; };
    static K make_k(double k) {
        const float h = (float)k;
        return make_float2(h, (float)(k - (double)h));
    }
    static double value(K k) { return (double)k.x + (double)k.y; }
    static V make_v(double re, double im) {
        const K a = make_k(re), b = make_k(im);
        const float2 h = make_float2(a.x, b.x), l = make_float2(a.y, b.y);
        V r;
        std::memcpy(&r.h, &h, 8);
        std::memcpy(&r.l, &l, 8);
        return r;
    }
    __device__ __forceinline__ static R expand(K k) { return R{dup2(k.x), dup2(k.y)}; }
    __device__ __forceinline__ static F one() { return make_double2(1.0, 0.0); }
    // v + k u: the product's high part exactly (its negative n, so that the
    // residual is one fused multiply-add), the cross terms in FP32, TwoSum
    __device__ __forceinline__ static V madd(const V& v, f2 kh, f2 kl, f2 nkh, const V& u) {
        const f2 n = mul2(nkh, u.h);
        f2 pl = fma2(kh, u.h, n);
        pl = fma2(kh, u.l, pl);
        pl = fma2(kl, u.h, pl);
        const f2 s = sub2(v.h, n);
        const f2 bb = sub2(s, v.h);
        const f2 e = sub2(sub2(v.h, sub2(s, bb)), add2(n, bb));
        return V{s, add2(v.l, add2(e, pl))};
    }
    __device__ __forceinline__ static void rot(V& a, V& b, const R& r) {
        const f2 nh = neg2(r.h), nl = neg2(r.l);
        const V p = madd(a, r.h, r.l, nh, b);
        b = madd(b, nh, nl, r.h, a);
        a = p;
    }
    __device__ __forceinline__ static V step(const V& v, K k, uint32_t minus, const V& u) {
        const R r = expand(minus ? make_float2(-k.x, -k.y) : k);
        return madd(v, r.h, r.l, neg2(r.h), u);
    }
    __device__ __forceinline__ static void norm(V& v) {
        const f2 h = add2(v.h, v.l);
        v.l = sub2(v.l, sub2(h, v.h));
        v.h = h;
    }
    __device__ __forceinline__ static V cmul(const V& w, const V& v) {
        const float2 wh = unpack2(w.h), wl = unpack2(w.l);
        const f2 rh = dup2(wh.x), rl = dup2(wl.x);
        V t;
        t.h = mul2(rh, v.h);
        t.l = fma2(rh, v.h, neg2(t.h));
        t.l = fma2(rh, v.l, t.l);
        t.l = fma2(rl, v.h, t.l);
        const f2 ih = pack2(-wh.y, wh.y), il = pack2(-wl.y, wl.y);
        V r = madd(t, ih, il, neg2(ih), V{swap2(v.h), swap2(v.l)});
        norm(r);
        return r;
    }
    __device__ __forceinline__ static V neg(const V& v, uint32_t odd) {
        const uint32_t s = odd << 31;
        const f2 m = ((f2)s << 32) | s;
        return V{v.h ^ m, v.l ^ m};
    }
    __device__ __forceinline__ static void ld(V& v, const V* p) {
        const ulonglong2 t = __ldcg(reinterpret_cast<const ulonglong2*>(p));
        v.h = t.x;
        v.l = t.y;
    }
};

struct BF64 {
    using V = double2;
    using K = double;
    static constexpr int kGroup = 3;
    static constexpr int kTiny = 7;
    static constexpr int kSw = 3;
    using R = double;
    static K make_k(double k) { return k; }
    static double value(K k) { return k; }
    static V make_v(double re, double im) { return make_double2(re, im); }
    using F = V;
    static F make_f(double re, double im) { return make_double2(re, im); }
    static double kept(double x) { return x; }
    __device__ __forceinline__ static F fmul(const F& a, const F& b) { return cmul(a, b); }
    __device__ __forceinline__ static V to_v(const F& f) { return f; }
    __device__ __forceinline__ static R expand(K k) { return k; }
    __device__ __forceinline__ static F one() { return make_double2(1.0, 0.0); }
    __device__ __forceinline__ static void rot(V& a, V& b, R k) {
        const V p = make_double2(__fma_rn(k, b.x, a.x), __fma_rn(k, b.y, a.y));
        b = make_double2(__fma_rn(-k, a.x, b.x), __fma_rn(-k, a.y, b.y));
        a = p;
    }
    __device__ __forceinline__ static V step(const V& v, K k, uint32_t minus, const V& u) {
        const double s = minus ? -k : k;
        return make_double2(__fma_rn(s, u.x, v.x), __fma_rn(s, u.y, v.y));
    }
    __device__ __forceinline__ static void norm(V&) {}
    __device__ __forceinline__ static V cmul(const V& w, const V& v) {
        return make_double2(__fma_rn(w.x, v.x, -__dmul_rn(w.y, v.y)), __fma_rn(w.x, v.y, __dmul_rn(w.y, v.x)));
    }
    __device__ __forceinline__ static V neg(const V& v, uint32_t odd) {
        const int s = (int)(odd << 31);
        return make_double2(__hiloint2double(__double2hiint(v.x) ^ s, __double2loint(v.x)),
                            __hiloint2double(__double2hiint(v.y) ^ s, __double2loint(v.y)));
    }
    __device__ __forceinline__ static void ld(V& v, const V* p) { v = __ldcg(p); }
};

// Energy sums of one thread: z += f |v|^2 (f a small integer), x += Re(conj(w) v).
// Packed float pairs with exact products (one lane of the pair per component)
// for FP32 and double-float, plain FP64 fused multiply-adds for FP64.
template <class P>
struct EAcc {
    f2 zs = 0, ze = 0, xs = 0, xe = 0;
    __device__ __forceinline__ static void high_low(const f2& v, f2& h, f2& l) { h = v; l = 0; }
    __device__ __forceinline__ static void high_low(const BDF::V& v, f2& h, f2& l) { h = v.h; l = v.l; }
    __device__ __forceinline__ static void prod(const typename P::V& w, const typename P::V& v, f2& h, f2& l) {
        f2 wh, wl, vh, vl;
        high_low(w, wh, wl);
        high_low(v, vh, vl);
        h = mul2(wh, vh);
        l = fma2(wh, vh, neg2(h));
        if (sizeof(typename P::V) == 16) {
            l = fma2(wh, vl, l);
            l = fma2(wl, vh, l);
        }
    }
    __device__ __forceinline__ void add_z(const typename P::V& v, float f) {
        f2 h, l, s, e;
        prod(v, v, h, l);
        const f2 ff = dup2(f);
        const f2 p = mul2(h, ff);
        const f2 pe = fma2(l, ff, fma2(h, ff, neg2(p)));
        two_sum(zs, p, s, e);
        zs = s;
        ze = add2(ze, add2(e, pe));
    }
    __device__ __forceinline__ void add_x(const typename P::V& w, const typename P::V& v) {
        f2 h, l, s, e;
        prod(w, v, h, l);
        two_sum(xs, h, s, e);
        xs = s;
        xe = add2(xe, add2(e, l));
    }
    __device__ __forceinline__ static double total(f2 s, f2 e) {
        const float2 a = unpack2(s), b = unpack2(e);
        return ((double)a.x + (double)b.x) + ((double)a.y + (double)b.y);
    }
    __device__ double z() const { return total(zs, ze); }
    __device__ double x() const { return total(xs, xe); }
};
template <>
struct EAcc<BF64> {
    double zs = 0.0, xs = 0.0;
    __device__ __forceinline__ void add_z(const double2& v, float f) {
        zs = __fma_rn(__fma_rn(v.x, v.x, __dmul_rn(v.y, v.y)), (double)f, zs);
    }
    __device__ __forceinline__ void add_x(const double2& w, const double2& v) {
        xs = __fma_rn(w.x, v.x, __fma_rn(w.y, v.y, xs));
    }
    __device__ double z() const { return zs; }
    __device__ double x() const { return xs; }
};

template <class P>
struct BatchArgs {
    typename P::V* states;
    const typename P::K* kap;      // kappa per (circuit, layer, qubit)
    const typename P::F* fac;      // factors per (circuit, layer, qubit, slot bit)
    const uint32_t* flips;         // per (circuit, layer): slot ^ logical
    const Item* items;
    const Circ* circ;
    int nitems;
    int T;
    int layers;
    double hx;
    unsigned* head;
    unsigned* counters;
    unsigned* status;      // nonzero: a wait timed out
    double2* partials;     // (zz sum, x sum) per energy slot
    double* energies;
    long long spin_limit;
};

// Shared-memory slot of tile element i: the lowest bits XORed with the next
// ones, so that both unit strides and the strides of the lowest register
// groups reach distinct banks (2^kSw elements fill the 32 banks).
template <class P>
__device__ __forceinline__ uint32_t slot(uint32_t i) {
    return i ^ ((i >> P::kSw) & ((1u << P::kSw) - 1u));
}

constexpr int kTabA = 64, kTabB = 128;   // table entries: local bits 0..5 and 6..12

// One tile as a pass sees it: local bits [0, nb) are qubits [0, L) and
// [hq, hq + nb - L); the tile index t holds the nt qubits from tq on.
struct Layout {
    int nb, L, hq, nt, tq;
    __device__ __forceinline__ int qubit(int j) const { return j < L ? j : hq + (j - L); }
    __device__ __forceinline__ uint32_t index(uint32_t l, uint32_t t) const {
        return (l & ((1u << L) - 1u)) | ((l >> L) << hq) | (t << tq);
    }
};

// Where a group's amplitudes come from and go to.
enum { kFromTile = 0, kFromGlobal = 1, kFromProduct = 2 };
enum { kToTile = 1, kToGlobal = 2 };

template <class P>
struct Group {
    typename P::V* tile;
    typename P::V* st;              // the circuit's HBM state (large circuits)
    const typename P::V *tabA, *tabB;   // the diagonal's (or product state's) tables
    const typename P::V* tf;        // factor of the tile's bits (null: none)
    Layout lay;
    uint32_t t;
    uint32_t flip;                  // slot ^ logical of the diagonal
    int src, dst;
    int diag;                       // multiply by the diagonal before writing
};

template <class P>
__device__ __forceinline__ uint32_t cz_odd(uint32_t x) { return (uint32_t)__popc(x & (x >> 1)) & 1u; }

// The factor of slot index l: tables, the tile's scalar and the CZ sign.
template <class P>
__device__ __forceinline__ typename P::V factor(const Group<P>& g, const typename P::V& w, uint32_t l) {
    const uint32_t x = g.lay.index(l, g.t) ^ g.flip;
    return P::neg(P::cmul(w, g.tabB[l >> 6]), cz_odd<P>(x));
}
template <class P>
__device__ __forceinline__ typename P::V factor_low(const Group<P>& g, uint32_t l) {
    const typename P::V a = g.tabA[l & 63u];
    return g.tf ? P::cmul(*g.tf, a) : a;
}

// The rotations of local bits b0 .. b0 + G - 1 (kappas k[0..G-1]; null: none)
// on the tile, in registers.
template <class P, int G>
__device__ void run_group(const Group<P>& g, int b0, const typename P::K* k) {
    using V = typename P::V;
    constexpr int E = 1 << G;
    typename P::R r[G];
    if (k) {
#pragma unroll
        for (int t = 0; t < G; ++t) r[t] = P::expand(k[t]);
    }
    const uint32_t below = (1u << b0) - 1u;
    const int nbase = 1 << (g.lay.nb - G);
    for (int b = threadIdx.x; b < nbase; b += blockDim.x) {
        const uint32_t base = (((uint32_t)b & ~below) << G) | ((uint32_t)b & below);
        V v[E];
        if (g.src == kFromTile) {
#pragma unroll
            for (int j = 0; j < E; ++j) v[j] = g.tile[slot<P>(base | ((uint32_t)j << b0))];
        } else if (g.src == kFromGlobal) {
#pragma unroll
            for (int j = 0; j < E; ++j) P::ld(v[j], g.st + g.lay.index(base | ((uint32_t)j << b0), g.t));
        } else {
#pragma unroll
            for (int j = 0; j < E; ++j) {
                const uint32_t l = base | ((uint32_t)j << b0);
                v[j] = factor<P>(g, factor_low<P>(g, l), l);
            }
        }
        if (k) {
#pragma unroll
            for (int t = 0; t < G; ++t)
#pragma unroll
                for (int j = 0; j < E; ++j)
                    if (!(j & (1 << t))) P::rot(v[j], v[j | (1 << t)], r[t]);
#pragma unroll
            for (int j = 0; j < E; ++j) P::norm(v[j]);
        }
        if (g.diag) {
            V w = factor_low<P>(g, base);
#pragma unroll
            for (int j = 0; j < E; ++j) {
                const uint32_t l = base | ((uint32_t)j << b0);
                if (j > 0 && b0 < 6) w = factor_low<P>(g, l);
                v[j] = P::cmul(factor<P>(g, w, l), v[j]);
            }
        }
        if (g.dst & kToTile) {
#pragma unroll
            for (int j = 0; j < E; ++j) g.tile[slot<P>(base | ((uint32_t)j << b0))] = v[j];
        }
        if (g.dst & kToGlobal) {
#pragma unroll
            for (int j = 0; j < E; ++j) g.st[g.lay.index(base | ((uint32_t)j << b0), g.t)] = v[j];
        }
    }
}

template <class P>
__device__ void run_group_n(const Group<P>& g, int size, int b0, const typename P::K* k) {
    switch (size) {
        case 4:
            if constexpr (P::kGroup >= 4) run_group<P, 4>(g, b0, k);
            break;
        case 3: run_group<P, 3>(g, b0, k); break;
        case 2: run_group<P, 2>(g, b0, k); break;
        default: run_group<P, 1>(g, b0, k); break;
    }
}

// The rotations of local bits [b0, b0 + cnt) (kappa k[i] for bit b0 + i), cnt
// >= 1, as register groups of at most kGroup bits.  top_first: the topmost
// group first (it reads global memory in contiguous runs), then the others
// upwards; else upwards.  `g` describes the first group's source and the last
// group's destination and diagonal; the groups in between use the tile.
template <class P>
__device__ void run_groups(Group<P> g, int b0, int cnt, const typename P::K* k, bool top_first) {
    const int ng = (cnt + P::kGroup - 1) / P::kGroup;
    const int dst = g.dst, diag = g.diag;
    for (int i = 0; i < ng; ++i) {
        const int m = top_first ? (i == 0 ? ng - 1 : i - 1) : i;
        // sizes cnt / ng, one more for the topmost ones
        const int q = cnt / ng, rem = cnt % ng;
        const int size = q + (m >= ng - rem ? 1 : 0);
        const int off = m * q + max(0, m - (ng - rem));
        g.dst = i == ng - 1 ? dst : kToTile;
        g.diag = i == ng - 1 ? diag : 0;
        run_group_n<P>(g, size, b0 + off, k + off);
        g.src = kFromTile;
        if (g.dst & kToTile) __syncthreads();
    }
}

// X terms of local bits [b0, b0 + G), and with `z` the ZZ terms.
template <class P, int G>
__device__ void energy_group(const Group<P>& g, int b0, bool z, int n, EAcc<P>& acc) {
    using V = typename P::V;
    constexpr int E = 1 << G;
    const uint32_t below = (1u << b0) - 1u;
    const uint32_t zmask = (n > 1) ? ((1u << (n - 1)) - 1u) : 0u;
    const int nbase = 1 << (g.lay.nb - G);
    for (int b = threadIdx.x; b < nbase; b += blockDim.x) {
        const uint32_t base = (((uint32_t)b & ~below) << G) | ((uint32_t)b & below);
        V v[E];
#pragma unroll
        for (int j = 0; j < E; ++j) {
            const uint32_t l = base | ((uint32_t)j << b0);
            if (g.src == kFromTile) v[j] = g.tile[slot<P>(l)];
            else P::ld(v[j], g.st + g.lay.index(l, g.t));
            if (g.dst & kToTile) g.tile[slot<P>(l)] = v[j];
        }
        if (z) {
#pragma unroll
            for (int j = 0; j < E; ++j) {
                const uint32_t x = g.lay.index(base | ((uint32_t)j << b0), g.t) ^ g.flip;
                acc.add_z(v[j], (float)((n - 1) - 2 * __popc((x ^ (x >> 1)) & zmask)));
            }
        }
#pragma unroll
        for (int t = 0; t < G; ++t)
#pragma unroll
            for (int j = 0; j < E; ++j)
                if (!(j & (1 << t))) acc.add_x(v[j | (1 << t)], v[j]);
    }
}

// X terms of local bits [b0, b0 + cnt), cnt >= 1; the topmost group first
// (from g.src, into the tile when other groups follow).
template <class P>
__device__ void run_energy(Group<P> g, int b0, int cnt, bool z, int n, EAcc<P>& acc) {
    const int ng = (cnt + 2) / 3;
    for (int m = ng - 1; m >= 0; --m) {
        const int q = cnt / ng, rem = cnt % ng;
        const int size = q + (m >= ng - rem ? 1 : 0);
        const int off = m * q + max(0, m - (ng - rem));
        g.dst = (m == ng - 1 && ng > 1 && g.src != kFromTile) ? kToTile : 0;
        switch (size) {
            case 3: energy_group<P, 3>(g, b0 + off, z, n, acc); break;
            case 2: energy_group<P, 2>(g, b0 + off, z, n, acc); break;
            default: energy_group<P, 1>(g, b0 + off, z, n, acc); break;
        }
        z = false;
        if (g.dst & kToTile) __syncthreads();
        g.src = kFromTile;
    }
}

template <class T>
__device__ __forceinline__ T shuffle_words(const T& v, uint32_t lane, bool flip) {
    T r;
    const uint32_t* s = reinterpret_cast<const uint32_t*>(&v);
    uint32_t* d = reinterpret_cast<uint32_t*>(&r);
#pragma unroll
    for (int k = 0; k < (int)(sizeof(T) / 4); ++k)
        d[k] = flip ? __shfl_xor_sync(0xffffffffu, s[k], lane) : __shfl_sync(0xffffffffu, s[k], lane);
    return r;
}

// Circuits of at most P::kTiny qubits: a warp each, amplitude x in lane x & 31 and
// register x >> 5, rotations of the low five qubits by shuffles, no barriers, the
// next layer's factors loaded ahead.  One CTA a circuit, its amplitudes in
// register groups, leaves most of its threads idle and waits at two barriers a
// layer: 2000 circuits of six qubits, 40 layers, complex64 535 -> 43 us,
// double-float 1187 -> 281, FP64 2052 -> 388 (368, 648 and 2098 a gate at a time); 256
// of four qubits, 8 layers, 39 -> 23, 46 -> 31 and 52 -> 31 (29, 40 and 64).
template <class P>
struct TinyArgs {
    const typename P::K* kap;
    const typename P::F* fac;
    const uint32_t* flips;
    const Circ* circ;
    const int* which;      // the circuits
    int count, layers;
    double hx;
    double* energies;
};

template <class P, int E>
__device__ void tiny_circuit(const TinyArgs<P>& a, int c) {
    using V = typename P::V;
    using F = typename P::F;
    const Circ cc = a.circ[c];
    const int n = cc.n;
    const uint32_t lane = threadIdx.x & 31u;
    const bool in = lane < (1u << n);
    const uint32_t* flips = a.flips + cc.f_off;
    const F* fac = a.fac + 2 * cc.u_off;
    const typename P::K* kap = a.kap + cc.u_off;
    // the diagonal (of layer 0: the product state): products over qubits 0..3 in
    // lanes 0..15, over 4..7 in lanes 16..31
    const int q0 = lane < 16u ? 0 : 4, nf = max(0, min(4, n - q0));
    F f[4];
    typename P::K kl{};
    auto load = [&]() {
#pragma unroll
        for (int j = 0; j < 4; ++j) f[j] = j < nf ? fac[2 * (q0 + j) + ((lane >> j) & 1u)] : P::one();
        if ((int)lane < n) kl = kap[lane];
    };
    load();
    // the last qubits of the register groups that a CTA would make (run_groups),
    // where the amplitudes are renormalised
    uint32_t ends = 0;
    for (int m = 0, ng = (n + P::kGroup - 1) / P::kGroup, at = 0; m < ng; ++m) {
        at += n / ng + (m >= ng - n % ng ? 1 : 0);
        ends |= 1u << (at - 1);
    }
    V v[E];
    for (int l = 0; l < a.layers; ++l) {
        F w = f[0], mine[4];
#pragma unroll
        for (int j = 1; j < 4; ++j)
            if (j < nf) w = P::fmul(f[j], w);
#pragma unroll
        for (int j = 0; j < 4; ++j) mine[j] = f[j];
        const typename P::K kk = kl;
        fac += 2 * n;
        kap += n;
        if (l + 1 < a.layers) load();
        if (l > 0) {
            for (int q = 0; q < n; ++q) {
                const typename P::K k = shuffle_words(kk, (uint32_t)q, false);
                if (q < 5) {
#pragma unroll
                    for (int e = 0; e < E; ++e) v[e] = P::step(v[e], k, (lane >> q) & 1u, shuffle_words(v[e], 1u << q, true));
                } else {
                    const typename P::R r = P::expand(k);
#pragma unroll
                    for (int b = 1; b < E; b *= 2)
                        if (q == 5 + (b > 1) + (b > 2))
#pragma unroll
                            for (int e = 0; e < E; ++e)
                                if (!(e & b)) P::rot(v[e], v[e | b], r);
                }
                if (ends >> q & 1u) {
#pragma unroll
                    for (int e = 0; e < E; ++e) P::norm(v[e]);
                }
            }
        }
        const F low = shuffle_words(w, lane & 15u, false);
        const uint32_t flip = flips[l];
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const uint32_t x = lane | ((uint32_t)e << 5);
            const uint32_t y = x ^ flip;
            // in the order of the tables' products, which rounds alike
            F t = low;
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                const F h = shuffle_words(mine[j], 16u | (x >> 4 & (1u << j)), false);
                if (n > 4 + j) t = P::fmul(h, t);
            }
            V d = P::to_v(t);
            if (E > 2) {
                F h = shuffle_words(mine[2], 16u | (x >> 4 & 4u), false);
                const F h7 = shuffle_words(mine[3], 16u | (x >> 4 & 8u), false);
                if (n > 7) h = P::fmul(h7, h);
                d = P::cmul(d, P::to_v(h));
            }
            d = P::neg(d, cz_odd<P>(y & ((1u << n) - 1u)));
            v[e] = l == 0 ? d : P::cmul(d, v[e]);
        }
    }
    EAcc<P> acc;
    const uint32_t flip = flips[a.layers - 1], zmask = (1u << (n - 1)) - 1u;
#pragma unroll
    for (int e = 0; e < E; ++e) {
        const uint32_t x = (lane | ((uint32_t)e << 5)) ^ flip;
        if (in) acc.add_z(v[e], (float)((n - 1) - 2 * __popc((x ^ (x >> 1)) & zmask)));
        for (int q = 0; q < min(n, 5); ++q) {
            const V u = shuffle_words(v[e], 1u << q, true);
            if (in && !((lane >> q) & 1u)) acc.add_x(u, v[e]);
        }
#pragma unroll
        for (int b = 1; b < E; b *= 2)
            if (!(e & b)) acc.add_x(v[e | b], v[e]);
    }
    double z = acc.z(), x = acc.x();
    for (int o = 16; o > 0; o >>= 1) {
        z += __shfl_down_sync(0xffffffffu, z, o);
        x += __shfl_down_sync(0xffffffffu, x, o);
    }
    if (lane == 0) a.energies[c] = (z + 2.0 * a.hx * x) * cc.scale2;
}

constexpr int kTinyThreads = 128;
template <class P>
__global__ void __launch_bounds__(kTinyThreads) k_batch_tiny(const __grid_constant__ TinyArgs<P> a) {
    const int i = (int)((blockIdx.x * (unsigned)kTinyThreads + threadIdx.x) >> 5);
    if (i >= a.count) return;
    const int c = a.which[i], n = a.circ[c].n;
    if (n <= 5) tiny_circuit<P, 1>(a, c);
    else if (n == 6) tiny_circuit<P, 2>(a, c);
    else if (P::kTiny < 8 || n == 7) tiny_circuit<P, 4>(a, c);
    else if constexpr (P::kTiny >= 8) tiny_circuit<P, 8>(a, c);
}

// Partial products of the factors (2 per qubit) over the local bits 0..5 and
// 6..nb-1, and (by the last warp) the product over the tile's bits into *tf.
template <class P>
__device__ void build_tables(const Layout& lay, const typename P::F* fac, typename P::V* tabA, typename P::V* tabB) {
    const int na = lay.nb < 6 ? lay.nb : 6;
    const int ta = 1 << na, tb = 1 << (lay.nb - na);
    for (int i = threadIdx.x; i < ta + tb; i += blockDim.x) {
        const bool low = i < ta;
        const uint32_t e = low ? i : i - ta;
        const int j0 = low ? 0 : na, cnt = low ? na : lay.nb - na;
        typename P::F w = P::one();
        for (int j = 0; j < cnt; ++j) {
            const typename P::F f = fac[2 * lay.qubit(j0 + j) + ((e >> j) & 1u)];
            w = j == 0 ? f : P::fmul(f, w);
        }
        if (low) tabA[e] = P::to_v(w);
        else tabB[e] = P::to_v(w);
    }
}
template <class P>
__device__ void build_tile_factor(const Layout& lay, const typename P::F* fac, uint32_t t, typename P::V* tf) {
    const int last = (blockDim.x >> 5) - 1;
    if ((int)(threadIdx.x >> 5) != last) return;
    const int lane = threadIdx.x & 31;
    typename P::F w = lane < lay.nt ? fac[2 * (lay.tq + lane) + ((t >> lane) & 1u)] : P::one();
    for (int o = 1; o < lay.nt; o <<= 1) {
        typename P::F u;
        const uint32_t* s = reinterpret_cast<const uint32_t*>(&w);
        uint32_t* d = reinterpret_cast<uint32_t*>(&u);
#pragma unroll
        for (int k = 0; k < (int)(sizeof(w) / 4); ++k) d[k] = __shfl_xor_sync(0xffffffffu, s[k], o);
        w = P::fmul(u, w);
    }
    if (lane == 0) *tf = P::to_v(w);
}

// Block-wide sum; result valid in thread 0.
__device__ double block_sum(double d, double* sh) {
    for (int o = 16; o > 0; o >>= 1) d += __shfl_down_sync(0xffffffffu, d, o);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = d;
    __syncthreads();
    double tot = 0.0;
    if (threadIdx.x == 0)
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) tot += sh[w];
    return tot;
}

template <class P>
__global__ void __maxnreg__(128) k_batch(const __grid_constant__ BatchArgs<P> a) {
    using V = typename P::V;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    V* tile = reinterpret_cast<V*>(smem_raw);
    V* tabA = tile + (1u << a.T);
    V* tabB = tabA + kTabA;
    V* s_tf = tabB + kTabB;
    __shared__ double shred[32];
    __shared__ int s_item;
    __shared__ int s_ok;
    const int T = a.T;
    for (;;) {
        if (threadIdx.x == 0) s_item = (int)atomicAdd(a.head, 1u);
        __syncthreads();
        const int idx = s_item;
        __syncthreads();
        if (idx >= a.nitems) return;
        const Item it = a.items[idx];
        const Circ cc = a.circ[it.circuit];
        const int n = cc.n;
        // wait for the circuit's earlier passes (bounded)
        if (threadIdx.x == 0) {
            int ok = 1;
            if (it.dep > 0) {
                long long spins = 0;
                while (*((volatile unsigned*)&a.counters[it.circuit]) < it.dep) {
                    // give up after the limit, or at once if another wait already failed
                    if (++spins > a.spin_limit || *((volatile unsigned*)a.status) != 0u) {
                        ok = 0;
                        atomicExch(a.status, 1u);
                        break;
                    }
                    __nanosleep(256);
                }
                __threadfence();
            }
            s_ok = ok;
        }
        __syncthreads();
        if (!s_ok) continue;
        const typename P::K* kap = a.kap + cc.u_off;
        const typename P::F* fac = a.fac + 2 * cc.u_off;
        const uint32_t* flips = a.flips + cc.f_off;
        EAcc<P> acc;
        Group<P> g;
        g.tile = tile;
        g.st = a.states + cc.state_off;
        g.tabA = tabA;
        g.tabB = tabB;
        g.tf = nullptr;
        g.t = 0;
        if (it.kind == 0) {
            // ------------------------------------------------ small circuit
            g.lay = Layout{n, n, n, 0, 0};
            build_tables<P>(g.lay, fac, tabA, tabB);
            __syncthreads();
            g.flip = flips[0];
            g.src = kFromProduct;
            g.dst = kToTile;
            g.diag = 0;
            run_group<P, 1>(g, 0, nullptr);
            __syncthreads();
            g.src = kFromTile;
            g.diag = 1;
            for (int l = 1; l < a.layers; ++l) {
                build_tables<P>(g.lay, fac + (size_t)l * 2 * n, tabA, tabB);
                __syncthreads();
                g.flip = flips[l];
                run_groups<P>(g, 0, n, kap + (size_t)l * n, false);
            }
            run_energy<P>(g, 0, n, true, n, acc);
            const double z = block_sum(acc.z(), shred);
            const double x = block_sum(acc.x(), shred);
            if (threadIdx.x == 0) a.energies[it.circuit] = (z + 2.0 * a.hx * x) * cc.scale2;
            __syncthreads();
            continue;
        }
        // ---------------------------------------------------- large circuit
        const int L = 2 * T - n;                 // chunk bits of the high layout
        const bool high = it.kind == 2;
        g.lay = high ? Layout{T, L, T, T - L, L} : Layout{T, T, T, n - T, T};
        g.flip = flips[it.first ? 0 : it.layer];
        // the diagonal of a high pass, or layer 0's product state
        const int tab_layer = it.first ? 0 : it.layer;
        const bool tables = it.first || high;
        if (tables) build_tables<P>(g.lay, fac + (size_t)tab_layer * 2 * n, tabA, tabB);
        for (uint32_t t = it.tile0; t < it.tile1; ++t) {
            g.t = t;
            if (tables) {
                build_tile_factor<P>(g.lay, fac + (size_t)tab_layer * 2 * n, t, s_tf);
                __syncthreads();
                g.tf = s_tf;
            }
            g.src = it.first ? kFromProduct : kFromGlobal;
            g.dst = kToGlobal;
            g.diag = 0;
            if (it.kind == 1) {
                run_groups<P>(g, 0, T, kap + (size_t)it.layer * n, true);
            } else if (high) {
                if (it.last) g.dst |= kToTile;
                if (it.first) {                  // a single layer: the product state itself
                    run_group<P, 1>(g, 0, nullptr);
                    if (it.last) __syncthreads();
                } else {
                    g.diag = 1;
                    run_groups<P>(g, L, n - T, kap + (size_t)it.layer * n + T, false);
                }
                if (it.last) {
                    g.src = kFromTile;
                    run_energy<P>(g, L, n - T, true, n, acc);
                }
            } else {
                run_energy<P>(g, 0, T, false, n, acc);
            }
            __syncthreads();
        }
        if (it.slot >= 0) {
            const double z = block_sum(acc.z(), shred);
            const double x = block_sum(acc.x(), shred);
            if (threadIdx.x == 0) a.partials[it.slot] = make_double2(z, x);
        }
        // publish completion; the CTA that completes the circuit sums its energy
        if (threadIdx.x == 0) {
            __threadfence();
            const unsigned done = atomicAdd(&a.counters[it.circuit], 1u) + 1u;
            if (done == (unsigned)cc.nitems) {
                __threadfence();
                double zsum = 0.0, xsum = 0.0;
                for (int k = 0; k < cc.nslots; ++k) {
                    // written by other CTAs before their counter increments:
                    // read through L2 (bypassing this SM's L1)
                    const double2 p = __ldcg(&a.partials[cc.slot0 + k]);
                    zsum += p.x;
                    xsum += p.y;
                }
                a.energies[it.circuit] = (zsum + 2.0 * a.hx * xsum) * cc.scale2;
            }
        }
        __syncthreads();
    }
}

}  // namespace

}  // namespace qe

namespace qe {

namespace {

// Not inlined: compilers that contract a product and a sum into one rounding
// would break the error terms below.
__attribute__((noinline)) double rounded_product(double a, double b) { return a * b; }

// A product of sums of two squares in twice FP64's precision (hundreds of
// factors: FP64 roundings alone would add 5e-15).
struct Pair {
    double h = 1.0, l = 0.0;
    void times_squares(double a, double b) {
        const double aa = rounded_product(a, a), bb = rounded_product(b, b), s = aa + bb, t = s - aa;
        const double e = ((aa - (s - t)) + (bb - t)) + (std::fma(a, a, -aa) + std::fma(b, b, -bb));
        const double p = rounded_product(h, s), q = std::fma(h, s, -p) + (h * e + l * s);
        h = p + q;
        l = q - (h - p);
    }
};

// Host side of a layer: kappa, the slot factors and the flips of every
// rotation (see the top of the file), angles in qe_batch_create's order.
template <class P>
void upload_rotations(qe_batch* b, std::vector<uint64_t>& u_off, std::vector<double>& scale2) {
    u_off.resize(b->count);
    scale2.assign(b->count, 1.0);
    const size_t total = b->angles.size() / 2;
    std::vector<typename P::K> kap(total);
    std::vector<typename P::F> fac(2 * total);
    std::vector<uint32_t> flips((size_t)b->count * b->layers);
    size_t i = 0;
    for (int c = 0; c < b->count; ++c) {
        const int n = b->n[c];
        u_off[c] = i;
        uint32_t flip = 0;
        Pair norm;   // squared norm of the kept state, true state = kept / sqrt(norm)
        for (int l = 0; l < b->layers; ++l) {
            for (int q = 0; q < n; ++q, ++i) {
                const double th = b->angles[2 * i], ph = b->angles[2 * i + 1];
                const double cs = std::cos(0.5 * th);
                // in the slot basis a flipped qubit turns the other way
                const double sn = ((flip >> q) & 1u) ? -std::sin(0.5 * th) : std::sin(0.5 * th);
                const bool trade = std::fabs(sn) > std::fabs(cs);
                kap[i] = P::make_k(trade ? cs / sn : -sn / cs);
                const double k = P::value(kap[i]);
                if (trade) flip ^= 1u << q;
                // signs of slots 0 and 1: those of (c, c), or of (s, -s) when traded
                double f0 = std::copysign(1.0, trade ? sn : cs), f1 = trade ? -f0 : f0;
                if (l == 0) f1 *= -k;            // the product state: (p, q) of (1, 0)
                const double pc = std::cos(0.5 * ph), ps = std::sin(0.5 * ph);
                const double s0 = ((flip >> q) & 1u) ? ps : -ps;   // slot 0's logical bit is the flip
                // the squared norm's power of two, out of the layer's first factors
                double two = 1.0;
                if (q == 0 && std::isfinite(norm.h)) {
                    const int e = std::ilogb(norm.h) / 2;
                    two = std::ldexp(1.0, -e);
                    norm.h = std::ldexp(norm.h, -2 * e);
                    norm.l = std::ldexp(norm.l, -2 * e);
                }
                fac[2 * i] = P::make_f(two * f0 * pc, two * f0 * s0);
                fac[2 * i + 1] = P::make_f(two * f1 * pc, -two * f1 * s0);
                norm.times_squares(1.0, k);
                norm.times_squares(P::kept(pc), P::kept(ps));   // both slots' modulus
            }
            flips[(size_t)c * b->layers + l] = flip;
        }
        scale2[c] = 1.0 / norm.h;
    }
    const size_t fb = fac.size() * sizeof(fac[0]), kb = kap.size() * sizeof(kap[0]);
    if (b->fac) cudaFree(b->fac);
    b->fac = nullptr;
    QE_CUDA(cudaMalloc(&b->fac, fb + kb + flips.size() * sizeof(uint32_t)));
    b->kap = (char*)b->fac + fb;
    b->flips = (uint32_t*)((char*)b->kap + kb);
    QE_CUDA(cudaMemcpy(b->fac, fac.data(), fb, cudaMemcpyHostToDevice));
    QE_CUDA(cudaMemcpy(b->kap, kap.data(), kb, cudaMemcpyHostToDevice));
    QE_CUDA(cudaMemcpy(b->flips, flips.data(), flips.size() * sizeof(uint32_t), cudaMemcpyHostToDevice));
}

// States of the large circuits of one wave: together at most this many bytes.
// complex64 passes are short enough to want their states in L2 (half of its
// 129 MB: 25 ms for 512 circuits of 10..22 qubits, 28 ms with 256 MiB); the
// complex128 passes are bound by arithmetic and gain more from several large
// circuits that fill the gaps at the ends of each other's passes (with four
// tiles an item, double-float 72 against 92 ms, FP64 215 against 281 ms).
template <class P>
constexpr uint64_t kWaveBytes = (sizeof(typename P::V) == 16 ? 256ull : 64ull) << 20;

template <class P>
void build_plan(qe_batch* b) {
    const int T = b->plan.T;
    std::vector<uint64_t> u_off;
    std::vector<double> scale2;
    upload_rotations<P>(b, u_off, scale2);
    std::vector<Circ> circ(b->count);
    std::vector<Item> items;
    uint64_t state_off = 0;
    int slots = 0;
    std::vector<int> large;
    // Beside circuits of several passes the tiny ones fill the gaps between those
    // (200 circuits of 4..14 qubits 714 us as items, 722 beside).  Double-float: only
    // where there are no others (4..8 qubits 64.3 and 65.3 us), and with seven
    // qubits, which take a warp longer than a CTA, only where those outnumber the SMs
    const int largest = *std::max_element(b->n.begin(), b->n.end());
    int tiny_bits = largest > T ? 0 : P::kTiny;
    if (std::is_same<P, BDF>::value) {
        if (std::count(b->n.begin(), b->n.end(), P::kTiny) < 2 * num_sms()) --tiny_bits;
        if (largest > tiny_bits) tiny_bits = 0;
    }
    for (int c = 0; c < b->count; ++c) {
        Circ& cc = circ[c];
        cc.n = b->n[c];
        cc.u_off = u_off[c];
        cc.scale2 = scale2[c];
        cc.f_off = (uint64_t)c * b->layers;
        cc.state_off = 0;
        if (cc.n <= std::max(T, tiny_bits)) {
            cc.nitems = 1;
            cc.slot0 = 0;
            cc.nslots = 0;
        } else {
            cc.state_off = state_off;
            state_off += 1ull << cc.n;
            large.push_back(c);
        }
    }
    // large circuits largest first
    std::stable_sort(large.begin(), large.end(), [&](int x, int y) { return circ[x].n > circ[y].n; });
    // layer 0 is the product state that the first pass starts from
    const int P_ = b->layers > 1 ? 2 * (b->layers - 1) + 1 : 2;
    std::vector<std::vector<int>> per_pass_count(b->count, std::vector<int>(P_, 0));
    for (int c : large) {
        Circ& cc = circ[c];
        const uint32_t tiles = 1u << (cc.n - T);
        const uint32_t per = (uint32_t)std::max(1, b->plan.tiles_per_item);
        const int nper = (int)((tiles + per - 1) / per);
        cc.nitems = P_ * nper;
        cc.slot0 = slots;
        cc.nslots = 2 * nper;   // last high pass + energy low pass
        slots += cc.nslots;
    }
    size_t total_items = b->count;
    for (int c : large) total_items += circ[c].nitems;
    items.reserve(total_items);
    auto push_pass = [&](int c, int p) {
        const Circ& cc = circ[c];
        const uint32_t tiles = 1u << (cc.n - T);
        const uint32_t per = (uint32_t)std::max(1, b->plan.tiles_per_item);
        const int nper = (int)((tiles + per - 1) / per);
        for (int j = 0; j < nper; ++j) {
            Item it{};
            it.circuit = c;
            it.kind = (p == P_ - 1) ? 3 : (b->layers > 1 && p % 2 == 0) ? 1 : 2;
            it.layer = std::min(1 + p / 2, b->layers - 1);   // of the energy pass too: its flips are loaded
            it.first = p == 0;
            it.tile0 = j * per;
            it.tile1 = std::min(tiles, (uint32_t)(j + 1) * per);
            it.dep = (uint32_t)(p * nper);
            it.last = p == P_ - 2;
            it.slot = (p == P_ - 2) ? cc.slot0 + j : (p == P_ - 1) ? cc.slot0 + nper + j : -1;
            items.push_back(it);
        }
    };
    auto push_small = [&](int c) {
        Item it{};
        it.circuit = c;
        it.kind = 0;
        it.slot = -1;
        items.push_back(it);
    };
    // small circuits (largest first): one item each, without dependencies
    std::vector<int> small, tiny;
    for (int c = 0; c < b->count; ++c)
        if (circ[c].n <= tiny_bits) tiny.push_back(c);
        else if (circ[c].n <= T) small.push_back(c);
    std::stable_sort(small.begin(), small.end(), [&](int x, int y) { return circ[x].n > circ[y].n; });
    std::stable_sort(tiny.begin(), tiny.end(), [&](int x, int y) { return circ[x].n > circ[y].n; });
    // Large circuits go in waves (kWaveBytes: complex64 ones fit in the L2 cache,
    // so that a circuit's passes find its state there; complex128 ones exceed it
    // on purpose), pass-major inside a wave; the small circuits' items are spread evenly between
    // the passes, where they occupy CTAs that would otherwise wait for a
    // pass to finish.  Every item's dependencies (its circuit's earlier
    // passes) come earlier in this order, so the claimed items never wait on
    // unclaimed ones.
    std::vector<std::vector<int>> waves;
    uint64_t in_wave = 0;
    for (int c : large) {
        const uint64_t bytes = (1ull << circ[c].n) * sizeof(typename P::V);
        if (waves.empty() || in_wave + bytes > kWaveBytes<P>) {
            waves.emplace_back();
            in_wave = 0;
        }
        waves.back().push_back(c);
        in_wave += bytes;
    }
    const size_t gaps = waves.size() * (size_t)P_;
    size_t si = 0, gap = 0;
    for (const auto& w : waves)
        for (int p = 0; p < P_; ++p) {
            for (int c : w) push_pass(c, p);
            const size_t upto = small.size() * (++gap) / gaps;
            for (; si < upto; ++si) push_small(small[si]);
        }
    for (; si < small.size(); ++si) push_small(small[si]);
    // a layer indexes the flips, factors and kappas of the item's circuit
    for (const Item& it : items)
        if ((int)it.layer >= b->layers) fail(QE_ERR_STATE, "a batch work item names a layer beyond its circuit's last");
    b->nitems = (int)items.size();
    // device buffers
    const size_t need_states = state_off * sizeof(typename P::V);
    if (b->state_bytes < need_states) {
        if (b->states) cudaFree(b->states);
        b->states = nullptr;
        QE_CUDA(cudaMalloc(&b->states, std::max<size_t>(need_states, 256)));
        b->state_bytes = need_states;
    }
    if (b->items) cudaFree(b->items);
    if (b->circ) cudaFree(b->circ);
    if (b->tiny) cudaFree(b->tiny);
    b->tiny = nullptr;
    b->ntiny = (int)tiny.size();
    if (b->ntiny) {
        QE_CUDA(cudaMalloc(&b->tiny, tiny.size() * sizeof(int)));
        QE_CUDA(cudaMemcpy(b->tiny, tiny.data(), tiny.size() * sizeof(int), cudaMemcpyHostToDevice));
    }
    if (b->partials) cudaFree(b->partials);
    b->items = b->circ = nullptr;
    b->partials = nullptr;
    QE_CUDA(cudaMalloc(&b->items, std::max<size_t>(1, items.size()) * sizeof(Item)));
    QE_CUDA(cudaMemcpy(b->items, items.data(), items.size() * sizeof(Item), cudaMemcpyHostToDevice));
    QE_CUDA(cudaMalloc(&b->circ, circ.size() * sizeof(Circ)));
    QE_CUDA(cudaMemcpy(b->circ, circ.data(), circ.size() * sizeof(Circ), cudaMemcpyHostToDevice));
    QE_CUDA(cudaMalloc(&b->partials, std::max(1, slots) * sizeof(double2)));
    // algorithmic HBM bytes of one run: the first pass of a large circuit only
    // writes its state, the energy pass only reads it, the others do both:
    // 1 + 2 (P - 2) + 1 = 2 (P - 1) state sizes
    double bytes = 0.0;
    for (int c : large) bytes += 2.0 * (P_ - 1) * (double)((1ull << circ[c].n) * sizeof(typename P::V));
    b->hbm_bytes = bytes;
}

template <class P>
void capture(qe_batch* b) {
    if (b->exec) cudaGraphExecDestroy(b->exec);
    if (b->graph) cudaGraphDestroy(b->graph);
    b->exec = nullptr;
    b->graph = nullptr;
    static thread_local BatchArgs<P> a;
    a.states = reinterpret_cast<typename P::V*>(b->states);
    a.kap = reinterpret_cast<const typename P::K*>(b->kap);
    a.fac = reinterpret_cast<const typename P::F*>(b->fac);
    a.flips = b->flips;
    a.items = reinterpret_cast<const Item*>(b->items);
    a.circ = reinterpret_cast<const Circ*>(b->circ);
    a.nitems = b->nitems;
    a.T = b->plan.T;
    a.layers = b->layers;
    a.hx = b->hx;
    a.head = b->sync;
    a.status = b->sync + 1;
    a.counters = b->sync + 2;
    a.partials = b->partials;
    a.energies = b->energies;
    a.spin_limit = 1ll << 24;   // ~4 s of 256 ns sleeps
    const size_t smem = sizeof(typename P::V) * (((size_t)1 << b->plan.T) + kTabA + kTabB + 1);
    auto fn = k_batch<P>;
    QE_CUDA(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    int occ = 0;
    QE_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, fn, b->plan.threads, smem));
    if (occ < 1) fail(QE_ERR_UNSUPPORTED, "batch tile does not fit on an SM");
    const unsigned grid = (unsigned)std::min<long long>((long long)num_sms() * occ, b->nitems);
    cudaStream_t cs, ts = nullptr;
    cudaEvent_t fork = nullptr, join = nullptr;
    QE_CUDA(cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking));
    if (b->ntiny) {
        QE_CUDA(cudaStreamCreateWithFlags(&ts, cudaStreamNonBlocking));
        QE_CUDA(cudaEventCreateWithFlags(&fork, cudaEventDisableTiming));
        QE_CUDA(cudaEventCreateWithFlags(&join, cudaEventDisableTiming));
    }
    QE_CUDA(cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal));
    if (b->ntiny) {
        // a branch of its own: beside the others where they leave room
        TinyArgs<P> t;
        t.kap = a.kap;
        t.fac = a.fac;
        t.flips = a.flips;
        t.circ = a.circ;
        t.which = b->tiny;
        t.count = b->ntiny;
        t.layers = b->layers;
        t.hx = b->hx;
        t.energies = b->energies;
        cudaEventRecord(fork, cs);
        cudaStreamWaitEvent(ts, fork, 0);
        k_batch_tiny<P><<<(unsigned)((b->ntiny * 32ll + kTinyThreads - 1) / kTinyThreads), kTinyThreads, 0, ts>>>(t);
        cudaEventRecord(join, ts);
    }
    cudaMemsetAsync(b->sync, 0, (2 + b->count) * sizeof(unsigned), cs);
    if (grid > 0) fn<<<grid, b->plan.threads, smem, cs>>>(a);
    if (b->ntiny) cudaStreamWaitEvent(cs, join, 0);
    cudaMemcpyAsync(b->host_energies, b->energies, b->count * sizeof(double), cudaMemcpyDeviceToHost, cs);
    cudaMemcpyAsync(b->host_status, b->sync + 1, sizeof(unsigned), cudaMemcpyDeviceToHost, cs);
    cudaError_t e = cudaStreamEndCapture(cs, &b->graph);
    cudaStreamDestroy(cs);
    if (ts) cudaStreamDestroy(ts);
    if (fork) cudaEventDestroy(fork);
    if (join) cudaEventDestroy(join);
    QE_CUDA(e);
    QE_CUDA(cudaGraphInstantiate(&b->exec, b->graph, 0));
}

void prepare(qe_batch* b) {
    if (b->dtype == QE_C64) {
        build_plan<BF32>(b);
        capture<BF32>(b);
    } else if (b->arith == QE_ARITH_FP64) {
        build_plan<BF64>(b);
        capture<BF64>(b);
    } else {
        build_plan<BDF>(b);
        capture<BDF>(b);
    }
}

}  // namespace

void batch_create(qe_batch* b) {
    QE_CUDA(cudaMalloc(&b->sync, (2 + b->count) * sizeof(unsigned)));
    QE_CUDA(cudaMalloc(&b->energies, b->count * sizeof(double)));
    QE_CUDA(cudaMallocHost(&b->host_energies, b->count * sizeof(double)));
    QE_CUDA(cudaMallocHost(&b->host_status, sizeof(unsigned)));
    prepare(b);
}

void batch_run(qe_batch* b, double* out) {
    *b->host_status = 0;
    QE_CUDA(cudaGraphLaunch(b->exec, b->stream));
    QE_CUDA(cudaStreamSynchronize(b->stream));
    b->launches += 1;
    if (*b->host_status != 0) fail(QE_ERR_TIMEOUT, "a batch work item waited too long for its dependencies");
    if (out) std::copy(b->host_energies, b->host_energies + b->count, out);
}

void batch_set_arith(qe_batch* b, int arith) {
    b->arith = arith;
    prepare(b);
}

void batch_set_plan(qe_batch* b, int T, int tiles_per_item, int threads) {
    const int maxT = b->dtype == QE_C64 ? 13 : 12;
    int nmax = 0;
    for (int v : b->n) nmax = std::max(nmax, v);
    if (T < 4 || T > maxT || 2 * T - 1 < nmax) fail(QE_ERR_ARG, "tile bits out of range for this batch");
    if (tiles_per_item < 1 || (threads != 128 && threads != 256 && threads != 512)) fail(QE_ERR_ARG, "bad plan");
    b->plan.T = T;
    b->plan.tiles_per_item = tiles_per_item;
    b->plan.threads = threads;
    prepare(b);
}

void batch_destroy(qe_batch* b) {
    if (b->exec) cudaGraphExecDestroy(b->exec);
    if (b->graph) cudaGraphDestroy(b->graph);
    for (void* p : {b->states, b->fac, b->items, b->circ, (void*)b->tiny, (void*)b->sync, (void*)b->partials, (void*)b->energies})
        if (p) cudaFree(p);
    if (b->host_energies) cudaFreeHost(b->host_energies);
    if (b->host_status) cudaFreeHost(b->host_status);
}

}  // namespace qe
