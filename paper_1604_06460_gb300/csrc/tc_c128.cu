// Fused 5-qubit gates on complex128 states with the 5th-generation tensor
// cores: error-free integer-digit products on the FP16 tensor pipe (the
// splitting idea of Ozaki, Ogita, Oishi and Rump, "Error-free transformations
// of matrix multiplication by using fast routines of matrix multiplication
// and its applications", Numer. Algorithms 59, 2012), recombined exactly in
// 64-bit integers.
//
// A 5-qubit block acts on each group of 32 amplitudes (Sec. II, gate
// application); in real arithmetic a group is a 64-vector v = [Re x ; Im x]
// and the block is W = [[Re U, -Im U], [Im U, Re U]], so a tile of 128 groups
// is the product Out(128x64) = In(128x64) W^T.
//
// Two widths share the kernel, D = 7 digits (56-bit splitting, the FP64 mode)
// and D = 6 (48-bit splitting, the fast double-float mode).
//
// Splitting.  Row r of In (one group) is scaled by 2^(8D - E_r), where
// 2^(E_r - 1) bounds its largest magnitude, and every value becomes the
// integer X = round(|v| 2^(8D - E_r)) <= 2^(8D - 1), written in base 256 with
// balanced digits: X = sum_i a_i 256^(D - i), a_1 in [0, 128], a_2..a_D in
// [-128, 127]; the value's sign multiplies every digit.  Digit i thus weighs
// 2^(E_r - 8 i) whatever D is.  W's rows get scales 2^F_n and digits b_j the
// same way (by every CTA at its start).  Every digit is an integer of magnitude <= 128 and
// exact in FP16.
//
// Products.  C_d = sum_{i + j = d} A_i B_j^T for d = 2..D+2 (26 digit pairs
// for D = 6, 34 for D = 7), one FP32 tensor-memory accumulator per d; a pair
// with i + j = d carries units of 2^(E_r + F_n - 8 d).  One pair adds at most
// 64 * 128^2 = 2^20 units and no d has more than seven pairs, so every
// accumulator is an exact integer below 2^23, and those of d <= 5 (at most
// four pairs) lie in [-2^22, 2^22].
//
// Recombination (per output).  With the integer
//   Y = C_2 2^40 + C_3 2^32 + C_4 2^24 + C_5 2^16 + C_6 2^8
//       + round(C_7 + C_8 / 256 [+ C_9 / 65536 for D = 7]),
// |Y| < 2^61, the output is Y 2^(E_r + F_n - 56): one rounding of Y to a
// double plus an exact exponent shift.  C_2..C_5 become integers with the
// FP32 magic-number addition (C + 1.5 * 2^23 is exact for |C| <= 2^22 and its
// bit pattern minus that of 1.5 * 2^23 is C); C_6 and the last term with a
// float-to-integer conversion.
//
// Accuracy.  The splitting rounds each input to a multiple of 2^(E_r - 8D)
// and each matrix entry to one of 2^(F_n - 8D) (half a unit at most); the
// digit products are exact, the dropped pairs (i + j > D + 2) add at most
// 2^(E_r + F_n - 57.6) for D = 7 (2^(E_r + F_n - 50) for D = 6), and Y is
// rounded once.  Over the 64 terms of an output the input rounding adds at
// most 64 * 2^(E_r + F_n - 8D), so for D = 7 every output is within
// 2^(E_r + F_n - 50) of the exact product: inside the worst-case rounding
// error of an FP64 dot product of the same 64 terms (64 * 2^-53 * sum |v||w|,
// up to 2^(E_r + F_n - 41)), with 56-bit inputs (2^-56 of the row scale) where
// FP64 keeps 53 bits of each value.  D = 6 rounds inputs to 2^-48 of the row
// scale (bound 2^(E_r + F_n - 42)).  Rows whose largest magnitude is below
// 2^-920 are flushed to zero.
//
// Schedule (warp-specialised, one CTA per SM, persistent over tiles): eight
// warps split (four threads per group row), eight warps recombine (two per
// tensor-memory lane quarter), one warp issues the MMAs and two warps stream
// tiles in.  The 64 outputs of a row are computed as two halves of 32 (16
// complex columns each) into two tensor-memory accumulator sets X and Y.
// Per tile the MMAs run in the order X(real K), Y(real K), X(imaginary K),
// Y(imaginary K), so the digit slices are released in two parts: the
// splitters write the next tile's real-part digits as soon as both sets have
// consumed the current real parts, and its imaginary-part digits once the
// tile's last MMA is done.  The splitting of tile t + 1 (integer ALU work)
// thus overlaps the recombination of tile t (whose int64 -> double
// conversions run on the FP64 pipe), and a set is released to the MMAs as
// soon as its accumulators are in registers.  The staging buffer holds the
// raw amplitudes of a tile's half (64 group rows, column-major): two such
// buffers for D = 6, one for D = 7 (whose digit slices take the room of the
// second); the load warps refill a buffer with cp.async as soon as the
// splitters have read its half into registers (completion is signalled on the
// half's mbarrier), and prefetch the next tile into L2, a 128-byte line a
// lane (one bulk prefetch per contiguous run, 32 of them from one warp where
// all five qubits are high, held the loads up: 2.38 against 2.01 ms a pass on
// qubits 23..27 at n = 28).  The splitters derive each row's largest exponent from the
// values they hold.  Every hand-off is an mbarrier (count-based arrivals by
// threads, tcgen05.commit for MMA completion); waits suspend the thread until
// the phase completes, have an iteration limit, and on a timeout raise a
// shared abort flag that ends the waits of all other threads; the MMA warp
// waits for its own MMAs before tensor memory is freed.
#include <cmath>
#include <cstdlib>
#include <cstring>
#include <type_traits>

#include "qe_arith.cuh"
#include "qe_internal.h"
#include "qe_oz.cuh"
#include "qe_tc.cuh"

namespace qe {

namespace {

using namespace oz;
using tc::mbar_wait;
using tc::raise_status;
using tc::smem_u32;

constexpr int kEpiWarps = 8;                 // warps [0, 8): recombination, two per TMEM lane quarter
constexpr int kSplitWarps = 8;               // warps [8, 16): splitting, two threads per group row
constexpr int kLoadWarps = 2;                // one group row of each staged half per thread
constexpr int kSplitWarp0 = kEpiWarps, kMmaWarp = kEpiWarps + kSplitWarps, kLoadWarp0 = kMmaWarp + 1;
constexpr int kOzThreads = 32 * (kLoadWarp0 + kLoadWarps);   // 608: at most 5 warps per SM sub-partition
constexpr int kSplitThreads = 32 * kSplitWarps, kEpiThreads = 32 * kEpiWarps;
constexpr int kRows = 128;                    // groups per tile (MMA M)
constexpr int kK = 64;                        // real K
constexpr int kN = 64;                        // real N (two halves of 32)
constexpr int kNH = 32;                       // MMA N
constexpr uint32_t kTmemCols = 512;           // two accumulator sets of (D + 1) x 32 columns
constexpr uint32_t kSetY = 256;               // column of the second set
constexpr uint32_t kSliceA = kRows * 128;     // bytes of one digit slice of In (fp16, 128 B per row)
constexpr uint32_t kSliceB = kN * 128;        // bytes of one digit slice of W
constexpr int kHalfRows = kRows / 2;          // the staging buffer holds the two halves of a tile's rows,
constexpr uint32_t kHalfStage = kHalfRows * 32 * 16;   // each column-major: amplitude (row, column c) at 16 (64 c + row)
constexpr uint32_t kStackSlice = kNH * 128;   // bytes of one W' digit slice of one half (stacked along N)
constexpr int kFlushExp = 100;                // biased exponent below which a row is flushed

struct OzArgs {
    double2* x;
    uint64_t ntiles;
    int L, kh;
    uint8_t hq[12];
    uint8_t gpos[5];        // tile-local positions of the matrix bits, ascending
    uint32_t* status;
    long long spin_limit;
    int stall_test;         // failure-path test: the first staged half is never announced
};

// A block with its matrix (row-major), split into digits by every CTA.
struct GateArgs {
    OzArgs z;
    const double2* U;       // [32][32] in device memory (as a kernel parameter, read by lanes at different
                            // addresses, it cost 40 us a launch)
};

// One digit of a Fourier transform as a block whose matrix depends on `P` index
// bits outside the tile (see matrix_entry).
struct DftArgs {
    OzArgs z;               // z.hq the tile's bits at or above L
    int nskip;              // bits left out of a tile's index: the tile's and the P matrix bits, ascending
    uint8_t skip[32];
    int lt;                 // 2^lt tiles share a matrix
    int teams;              // CTAs i, i + teams, ... form team i; the matrices go to the teams in turn
    int P, vlo;             // the matrix bits [vlo, vlo + P)
    int d, below;           // the digit's bits, the idle matrix bits below them
    int reversed;           // leave the output bit-reversed in its qubits
    double scale;           // 2^(-d/2)
    const double2* roots;   // exp(+-2 pi i j / 2^(P + d)), j < 2^(P + d)
};

// mbarriers of the kernel
enum Bar {
    kReReady,     // splitters: real-part digits of the tile written (256 arrivals)
    kImReady,     // splitters: imaginary-part digits written (256)
    kReFree,      // commit: the MMAs over the real-part digits are done
    kXFull,       // commit: set X holds the tile's first half
    kYFull,       // commit: set Y holds the second half; all digits consumed
    kXFree,       // recombiners: set X read into registers (256)
    kYFree,       // recombiners: set Y read (256)
    kStage0,      // load warps: rows [0, 64) of the tile staged (64 cp.async arrivals)
    kStage1,      // rows [64, 128) staged
    kStageFree0,  // splitters: staged half 0 read (256)
    kStageFree1,  // staged half 1 read
    kEt0,         // splitters: row scales of the tile, ring slot 0 / 1 (128)
    kEt1,
    kDrain,       // commit: every MMA issued has completed
    kBars
};

// The MMA-issuing warp: all lanes compute the (warp-uniform) operands, one
// elected lane issues, so that the descriptors come from uniform registers
// (2.47 against 2.40 ms a pass at n = 28 with one divergent lane doing both:
// the kernel's period runs through this warp).  The accumulators of one half lie side by side,
// C_d at column 32 (d - 2), and each half's W' digit slices are stacked along
// N (rows 32 (j - 1) + m), so one MMA of A_i against the stacked slices
// j0..j1 writes C_{i + j0} .. C_{i + j1} at once: the digit products form a
// convolution (D = 6: 26 pairs in 7 MMAs per K-step and half; D = 7: 34 in
// 8).  Per tile: both halves' K-steps over the real parts (each half once
// its set is free), a commit that releases the real-part digits, then the
// imaginary-part K-steps of X (committed: X full) and of Y (committed: Y
// full and every digit consumed).
// `ph` holds the barrier phases across calls (bit 0 digits ready, bit 1 sets
// free, bit 2 no tile yet: 4 before the first call), bit 3 of the result that
// a wait ran out.
template <int D>
__device__ __forceinline__ uint32_t issue_mmas(uint32_t elected, const OzArgs& a, uint32_t t0, uint32_t t1,
                                               uint32_t step, uint32_t tmem, uint32_t a0, uint32_t b0, uint64_t* bars,
                                               uint32_t* abort_flag, uint32_t ph) {
    constexpr MmaTable<D> tab;
    constexpr uint32_t kStackB = (uint32_t)D * kStackSlice;
    const uint64_t da0 = tc::sdesc_sw128(a0);      // an offset of b bytes adds b >> 4
    auto issue = [&](int hh, int ks0, int ks1) {
        const uint32_t set = tmem + (hh ? kSetY : 0u);
        const uint64_t db0 = tc::sdesc_sw128(b0 + (uint32_t)hh * kStackB);
#pragma unroll
        for (int ks = 0; ks < kK / 16; ++ks) {
            if (ks < ks0 || ks >= ks1) continue;
#pragma unroll
            for (int m = 0; m <= D; ++m) {
                const int i = tab.i[m], j0 = tab.j0[m], j1 = tab.j1[m];
                const uint32_t nn = (uint32_t)(j1 - j0 + 1) * kNH;
                const uint64_t da = da0 + (((uint32_t)(i - 1) * kSliceA + 32u * ks) >> 4);
                const uint64_t db = db0 + (((uint32_t)(j0 - 1) * kStackSlice + 32u * ks) >> 4);
                const uint32_t dt = set + (uint32_t)(i + j0 - 2) * kNH;
                mma_f16_elected(elected, dt, da, db, tc::idesc(0u, nn, kRows), (ks > 0 || m > 1) ? 1u : 0u);
            }
        }
    };
    auto wait = [&](Bar b, uint32_t& ph) {
        const bool ok = wait_or_abort(smem_u32(&bars[b]), ph, a.spin_limit, abort_flag);
        if (__any_sync(0xFFFFFFFFu, !ok)) return false;
        ph ^= 1u;
        asm volatile("tcgen05.fence::after_thread_sync;");
        return true;
    };
    uint32_t pre = ph & 1u, pim = pre, pxf = (ph >> 1) & 1u, pyf = pxf;
    bool first = ph & 4u;
    for (uint32_t t = t0; t < t1; t += step) {
        if (!wait(kReReady, pre)) return 8u;
        if (!first && !wait(kXFree, pxf)) return 8u;
        issue(0, 0, 2);
        if (!first && !wait(kYFree, pyf)) return 8u;
        issue(1, 0, 2);
        mma_commit_elected(elected, &bars[kReFree]);
        if (!wait(kImReady, pim)) return 8u;
        issue(0, 2, 4);
        mma_commit_elected(elected, &bars[kXFull]);
        issue(1, 2, 4);
        mma_commit_elected(elected, &bars[kYFull]);
        first = false;
    }
    return pre | (pxf << 1) | (first ? 4u : 0u);
}

// Entry (row, column) of the block's complex matrix.
__device__ __forceinline__ double2 matrix_entry(const GateArgs& g, uint32_t, uint32_t row, uint32_t col) {
    return g.U[32 * row + col];
}
// Of a transform digit: with l_prior the P-bit value of the transform's outputs
// so far (the matrix bits v, which hold it bit-reversed),
//   U[l][k] = 2^(-d/2) w_(2^(P + d))^(k (l_prior + 2^P l)):
// the digit's 2^d-point transform with the twiddle by the earlier outputs
// folded into the columns.  With several digits, output l is left at the
// bit-reversed position, so that one bit reversal of the register restores the
// natural order whatever the digits are.
__device__ __forceinline__ double2 matrix_entry(const DftArgs& f, uint32_t v, uint32_t row, uint32_t col) {
    const uint32_t lp = f.P ? (__brev(v) >> (32 - f.P)) : 0u, dm = (1u << f.d) - 1u;
    const uint32_t lr = (row >> f.below) & dm, k = (col >> f.below) & dm;
    const uint32_t l = f.reversed ? __brev(lr) >> (32 - f.d) : lr;
    const double2 w = f.roots[(k * (lp + (l << f.P))) & ((1u << (f.P + f.d)) - 1u)];
    const bool inside = ((col ^ row) & ~(dm << f.below)) == 0;    // idle qubits: the identity
    return inside ? make_double2(w.x * f.scale, w.y * f.scale) : make_double2(0.0, 0.0);
}

// The digits and row scales of W = [[Re U, -Im U], [Im U, Re U]] in shared
// memory, by all warps: one warp per complex row, lane <-> column, every entry
// split like the inputs with the scale of its row's largest component (real
// rows n and n + 32 share it); rows below 2^-920 are flushed to zero.
template <int D, class Args>
__device__ __noinline__ void build_w(const Args& g, uint32_t v, unsigned char* sB, int* sF20) {
    constexpr uint32_t kStackB = (uint32_t)D * kStackSlice;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int r = warp; r < 32; r += kOzThreads / 32) {
        const double2 u = matrix_entry(g, v, (uint32_t)r, (uint32_t)lane);
        uint32_t em = max((uint32_t)__double2hiint(u.x) << 1, (uint32_t)__double2hiint(u.y) << 1);
        for (int o = 16; o > 0; o >>= 1) em = max(em, __shfl_xor_sync(0xFFFFFFFFu, em, o));
        em >>= 21;
        const uint32_t base_s = em < (uint32_t)kFlushExp ? 0x10000u : (D == 7 ? em : em + 5u);
        uint32_t dg[D];   // (re, im) digits as fp16 pairs
        digit_pairs<D>(split_z<D>(u.x, base_s), split_z<D>(u.y, base_s), dg);
        const int hh = r >> 4, m = r & 15;
        unsigned char* const b = sB + hh * kStackB + 2 * (lane & 7);
        const int c0 = lane >> 3, c1 = 4 + (lane >> 3);
#pragma unroll
        for (int j = 0; j < D; ++j) {
            const uint16_t dr = (uint16_t)dg[j], di = (uint16_t)(dg[j] >> 16);
            *reinterpret_cast<uint16_t*>(b + sw128_chunk(j * kNH + m, c0)) = dr;
            *reinterpret_cast<uint16_t*>(b + sw128_chunk(j * kNH + m, c1)) = di ^ 0x8000u;
            *reinterpret_cast<uint16_t*>(b + sw128_chunk(j * kNH + m + 16, c0)) = di;
            *reinterpret_cast<uint16_t*>(b + sw128_chunk(j * kNH + m + 16, c1)) = dr;
        }
        if (lane == 0) sF20[r] = sF20[32 + r] = em < (uint32_t)kFlushExp ? 0 : ((int)em - 1021) * (1 << 20);
    }
}

// Dynamic shared memory: D digit slices of In, D of W' (two stacked halves),
// and two staging buffers (D = 6) or one (D = 7), plus 1 KB of alignment.
template <int D>
constexpr size_t oz_smem() {
    return 1024 + (size_t)D * (kSliceA + kSliceB) + (D == 7 ? 1 : 2) * (size_t)kHalfStage;
}
static_assert(oz_smem<6>() <= 227 * 1024 && oz_smem<7>() <= 227 * 1024, "shared memory per CTA");

// Blocks with qubit 0 (PAIR: matrix bit 0 is qubit 0, so that columns 2j and
// 2j + 1 are neighbours in memory) load along memory instead of along rows and
// store 32 bytes at a time: qubits 0, 1, 2, 20, 27 at n = 28 took 3.43 ms a pass
// with a row a lane and 16-byte stores, 2.53 ms so; the other blocks do without
// the index arithmetic (2.04 against 2.08 ms).
// Byte offset of amplitude (row of 64, column c) in a staged half with PAIR:
// column-major, the rows of a column XORed with the reversal of the column's low three bits,
// so that the eight lanes of a 16-byte access reach different banks whether
// their index bits are row bits (low ones), column bits or some of each.  XOR
// linear in (row, column).
__host__ __device__ constexpr uint32_t stage_swizzle(uint32_t c) { return ((c & 1u) << 2) | (c & 2u) | ((c >> 2) & 1u); }
__device__ __forceinline__ uint32_t stage_off(uint32_t row, uint32_t c) {
    return 16u * (kHalfRows * c + (row ^ stage_swizzle(c)));
}

__device__ __forceinline__ const OzArgs& oz_args(const GateArgs& a) { return a.z; }
__device__ __forceinline__ const OzArgs& oz_args(const DftArgs& a) { return a.z; }

// The exponent term of a row whose largest biased exponent is em.
__host__ __device__ constexpr int eterm_of(int em) { return (em - 1021 - 56) * (1 << 20); }
constexpr int kEtermBad = eterm_of(0x7FF);

// 19 warps of 96 registers a thread: a sub-partition holding five of the warps
// uses 15,360 of its 16,384 registers (104 would exceed them).
//
// Without DFT, one matrix for all tiles, tile t = block, block + grid, ...
// With it, the 2^lt tiles of one matrix are a segment of a team of CTAs, each
// of which takes every step-th tile; between segments all roles meet at a
// barrier, build the next matrix and go on with their barrier phases.
template <int D, bool PAIR, class Args>
__global__ void __maxnreg__(96) k_gate_tc5_c128(const __grid_constant__ Args arg) {
    constexpr bool kDft = std::is_same<Args, DftArgs>::value;
    const OzArgs& a = oz_args(arg);
    constexpr int kAcc = D + 1;                  // accumulators C_2 .. C_{D+2}
    constexpr bool kOneStage = D == 7;           // one staging buffer for both halves of a tile
    constexpr uint32_t kStackB = (uint32_t)D * kStackSlice;
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char* base = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
    unsigned char* sA = base;                                   // D digit slices of In
    unsigned char* sB = sA + D * kSliceA;                       // per half: the D W' digit slices stacked
    unsigned char* stage = sB + D * kSliceB;                    // raw amplitudes of one or two tile halves
    __shared__ __align__(8) uint64_t bars[kBars];
    __shared__ uint32_t tmem_base, abort_flag;
    __shared__ uint64_t hoff[kDft ? 512 : 32];
    __shared__ uint32_t cpos[32];
    __shared__ uint64_t coloff[32];
    __shared__ ulonglong2 k_off[32];           // the loaders' k-th copy: offsets in memory and in the staging buffer
    __shared__ int sF20[kN];
    __shared__ int s_eterm[2][kRows];          // (E_r - 56) << 20 of the rows of two tiles in flight
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

    if constexpr (!kDft) build_w<D>(arg, 0u, sB, sF20);
    if (tid < (1 << a.kh)) {
        uint64_t o = 0;
        for (int j = 0; j < a.kh; ++j)
            if ((tid >> j) & 1) o |= 1ull << a.hq[j];
        hoff[tid] = o;
    }
    if (tid < 32) {
        uint32_t o = 0;
        for (int j = 0; j < 5; ++j)
            if ((tid >> j) & 1) o |= 1u << a.gpos[j];
        cpos[tid] = o;
    }
    if (tid == 0) {
        const uint32_t counts[kBars] = {kSplitThreads, kSplitThreads, 1,      1, 1, kEpiThreads, kEpiThreads,
                                        32 * kLoadWarps, 32 * kLoadWarps, kSplitThreads, kSplitThreads,
                                        kRows,         kRows,         1};
        for (int b = 0; b < kBars; ++b) mbar_init_count(&bars[b], counts[b]);
        abort_flag = 0u;
        asm volatile("fence.mbarrier_init.release.cluster;");
    }
    if (warp == kMmaWarp) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base)),
                     "r"(kTmemCols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    asm volatile("fence.proxy.async.shared::cta;");
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
    if (tid < 32) {
        const uint32_t l = cpos[tid];
        coloff[tid] = 16ull * ((l & ((1u << a.L) - 1u)) + hoff[l >> a.L]);   // bytes
    }
    __syncthreads();
    const uint32_t tmem = tmem_base;

    const uint32_t gmask = cpos[31];
    // tile-local row r (a group) <-> index bits: the seven non-gate local bits
    auto row_bits = [&](int r) {
        uint32_t l = 0;
        int j = 0;
        for (int b = 0; b < 12; ++b)
            if (!((gmask >> b) & 1u)) l |= (((uint32_t)r >> (j++)) & 1u) << b;
        return l;
    };
    auto row_off = [&](int r) {   // bytes
        const uint32_t l = row_bits(r);
        return 16ull * ((l & ((1u << a.L) - 1u)) + hoff[l >> a.L]);
    };
    // row (of 64) and column of the half's index whose lowest six bits in memory
    // order are i and whose others are k
    auto half_index = [&](uint32_t i, uint32_t k, uint32_t& row, uint32_t& col) {
        uint32_t rest = i | (k << 6), rb = 0, cb = 0;
        row = col = 0;
        for (int b = 0; b < 12 && rb + cb < 11; ++b) {
            if ((gmask >> b) & 1u) col |= (rest & 1u) << cb++;
            else if (rb < 6) row |= (rest & 1u) << rb++;
            else continue;
            rest >>= 1;
        }
    };
    if (PAIR && tid < 32) {
        uint32_t r, c;
        half_index(0, tid, r, c);
        k_off[tid] = make_ulonglong2(row_off(r) + coloff[c], stage_off(r, c));
    }
    __syncthreads();
    char* const xb = reinterpret_cast<char*>(a.x);
    auto tile_ptr = [&](uint32_t t) {
        if constexpr (kDft) {
            const uint64_t u = t & ((1u << arg.lt) - 1u), v = t >> arg.lt;
            return xb + 16ull * (insert_zero_bits(u << a.L, arg.skip, arg.nskip) | (v << arg.vlo));
        } else {
            return xb + 16ull * insert_zero_bits((uint64_t)t << a.L, a.hq, a.kh);
        }
    };
    // The CTA's current segment: tiles [begin, end) in steps of `step` (32 bits
    // hold any tile index).  With kDft they live in shared memory, where they
    // cost the roles no registers (the digit kernel spilled with them in
    // registers: 12.3 against 11.3 ms a pass at n = 30).
    __shared__ uint32_t s_begin, s_end, s_step, s_matrix;
    auto seg_begin = [&]() -> uint32_t { return kDft ? s_begin : blockIdx.x; };
    auto seg_end = [&]() -> uint32_t { return kDft ? s_end : (uint32_t)a.ntiles; };
    auto seg_step = [&]() -> uint32_t { return kDft ? s_step : gridDim.x; };
    // Starts the next segment (all threads): false when there is none or a
    // wait has run out.  The barrier before the rebuild follows the
    // recombination of the segment's last tile, hence all its MMAs.
    auto next_segment = [&](bool begin) {
        if constexpr (!kDft) {
            return begin;
        } else {
            const uint32_t team = blockIdx.x % arg.teams;
            uint32_t v = team;
            if (!begin) {
                __syncthreads();
                if (*reinterpret_cast<volatile uint32_t*>(&abort_flag)) return false;
                v = s_matrix + arg.teams;   // (not from s_begin: a CTA's place in its team may reach 2^lt)
                __syncthreads();
            }
            if (v >> arg.P) return false;
            if (tid == 0) {
                s_matrix = v;
                s_begin = (v << arg.lt) + blockIdx.x / arg.teams;
                s_end = (v + 1) << arg.lt;
                s_step = (gridDim.x - team + arg.teams - 1) / arg.teams;    // CTAs of the team
            }
            build_w<D>(arg, v, sB, sF20);
            asm volatile("fence.proxy.async.shared::cta;");
            __syncthreads();
            return true;
        }
    };
    // wait (all lanes of a warp) for a phase of barrier b; on a timeout or an
    // abort raise the status word.  The outcome is the same on every lane,
    // so the warp stays converged for its .sync.aligned instructions.
    auto wait = [&](Bar b, uint32_t& ph) {
        const bool ok = wait_or_abort(smem_u32(&bars[b]), ph, a.spin_limit, &abort_flag);
        if (__any_sync(0xFFFFFFFFu, !ok)) {
            if (!ok) raise_status(a.status);
            return false;
        }
        ph ^= 1u;
        return true;
    };
    if (warp == kMmaWarp) {
        // ---------------------------------------------------- MMA issuer
        uint32_t ph = 4u;
        const uint32_t elected = elect_lane();
        for (bool more = next_segment(true); more; more = next_segment(false)) {
            ph = issue_mmas<D>(elected, a, seg_begin(), seg_end(), seg_step(), tmem, smem_u32(sA), smem_u32(sB), bars,
                               &abort_flag, ph);
            if (ph & 8u) raise_status(a.status);
            __syncwarp();
        }
        mma_commit_elected(elected, &bars[kDrain]);    // by the lane that issued the MMAs
        if (lane == 0) {
            // every MMA issued has completed before tensor memory is freed
            if (!tc::mbar_wait(smem_u32(&bars[kDrain]), 0u, a.spin_limit)) raise_status(a.status);
        }
        __syncwarp();
    } else if (warp >= kLoadWarp0) {
        // ------------------------------------------------------- tile loads
        // per half, once the splitters have read it, 32 16-byte copies a thread
        // into the column-major staging buffer and an arrival on the half's
        // stage barrier when they land.  Thread <-> group row i of the half and
        // copy <-> column; with PAIR the half's 11 index bits (6 of the row, 5
        // of the column) are taken in the order of their place in memory, the
        // thread index holding the lowest six, so that a warp copies whole
        // lines where a row a lane would take 16-byte pieces
        const int i = tid - kLoadWarp0 * 32;
        uint32_t ri = i, ci = 0;
        if constexpr (PAIR) half_index(i, 0, ri, ci);
        const uint64_t go = row_off(ri) + coloff[ci], go_half = row_off(kHalfRows);
        const uint32_t so = PAIR ? stage_off(ri, ci) : 16u * ri;
        const uint32_t d = smem_u32(stage);
        uint32_t pf[2] = {0u, 0u};
        bool first = true, ok = true;
        for (bool more = next_segment(true); more; more = next_segment(false))
        for (uint32_t t = seg_begin(); t < seg_end() && ok; t += seg_step()) {
            const char* g = tile_ptr(t);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                // the buffer's previous half must have been read: with two
                // buffers the same half of the previous tile, with one the
                // other half (of this tile for h = 1, of the previous for h = 0)
                const int fh = kOneStage ? 1 - h : h;
                if (!(first && (h == 0 || !kOneStage)) && !wait(fh ? kStageFree1 : kStageFree0, pf[fh])) {
                    ok = false;
                    break;
                }
                const char* gr = g + go + (h ? go_half : 0ull);
                const uint32_t dh = d + (kOneStage ? 0u : (uint32_t)h * kHalfStage);
                if constexpr (PAIR) {
#pragma unroll 8
                    for (int k = 0; k < 32; ++k) {
                        const ulonglong2 o = k_off[k];
                        cp_async16(dh + (so ^ (uint32_t)o.y), gr + o.x);
                    }
                } else {
#pragma unroll 8
                    for (int c = 0; c < 32; ++c) cp_async16(dh + so + 16u * kHalfRows * c, gr + coloff[c]);
                }
                if (!(a.stall_test && first && h == 0)) cp_async_arrive(&bars[h ? kStage1 : kStage0]);
            }
            first = false;
            // the tile after this one into L2 meanwhile, a 128-byte line at a time
            // (2^(L-3) lines in each of its 2^kh runs)
            const uint32_t tn = t + seg_step();
            if (ok && tn < seg_end()) {
                const char* gn = tile_ptr(tn);
#pragma unroll
                for (int k = 0; k < 512 / (32 * kLoadWarps); ++k) {
                    const int l = i + 32 * kLoadWarps * k;
                    const char* gl = gn + 16ull * hoff[l >> (a.L - 3)] + 128u * (uint32_t)(l & ((1 << (a.L - 3)) - 1));
                    asm volatile("prefetch.global.L2 [%0];" ::"l"(gl) : "memory");
                }
            }
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
    } else if (warp >= kSplitWarp0) {
        // -------------------------------------------------------- splitting
        // thread <-> (row 64 h + ri of each half h, complex columns
        // [8 qq, 8 qq + 8)); the four threads of a row are lanes l, l ^ 8,
        // l ^ 16, l ^ 24 of one warp.  Per half: the 8 amplitudes into
        // registers (the staging half is then released), the row's largest
        // exponent by two shuffles, the real-part digits (operand chunk qq),
        // then the imaginary-part digits (chunk 4 + qq).
        const int sw = warp - kSplitWarp0;
        const int ri = 8 * sw + (lane & 7), qq = lane >> 3;
        const unsigned char* const scol = stage + 16u * kHalfRows * 8 * qq;   // column 8 qq
        uint32_t prf = 0, pyf = 0;
        bool first = true, ok = true;
        int it = 0;
        for (bool more = next_segment(true); more; more = next_segment(false))
        for (uint32_t t = seg_begin(); t < seg_end() && ok; t += seg_step(), ++it) {
            const uint32_t ph = (uint32_t)it & 1u;    // each stage barrier completes once per tile
#pragma unroll 1
            for (int h = 0; h < 2; ++h) {
                uint32_t phh = ph;
                if (!wait(h ? kStage1 : kStage0, phh)) {
                    ok = false;
                    break;
                }
                const int r = kHalfRows * h + ri;
                double2 v[8];
                const double2* src =
                    reinterpret_cast<const double2*>(scol + (kOneStage ? 0u : (uint32_t)h * kHalfStage));
#pragma unroll
                for (int k = 0; k < 8; ++k) v[k] = src[kHalfRows * k + (PAIR ? ri ^ (int)stage_swizzle(k) : ri)];
                mbar_arrive(&bars[h ? kStageFree1 : kStageFree0]);
                uint32_t em = 0;    // largest (high word << 1): the biased exponent in the top 11 bits
#pragma unroll
                for (int k = 0; k < 8; ++k)
                    em = max(em, max((uint32_t)__double2hiint(v[k].x) << 1, (uint32_t)__double2hiint(v[k].y) << 1));
                em = max(em, __shfl_xor_sync(0xFFFFFFFFu, em, 8));
                em = max(em, __shfl_xor_sync(0xFFFFFFFFu, em, 16));
                em >>= 21;
                const uint32_t base_s = (em < (uint32_t)kFlushExp) ? 0x10000u : (D == 7 ? em : em + 5u);
#pragma unroll
                for (int part = 0; part < 2; ++part) {
                    uint32_t w[D][4];            // packed fp16 pairs: slice i, values 2p, 2p + 1
#pragma unroll
                    for (int p2 = 0; p2 < 4; ++p2) {
                        const double2 va = v[2 * p2], vb = v[2 * p2 + 1];
                        uint32_t dg[D];
                        digit_pairs<D>(split_z<D>(part ? va.y : va.x, base_s), split_z<D>(part ? vb.y : vb.x, base_s),
                                       dg);
#pragma unroll
                        for (int k = 0; k < D; ++k) w[k][p2] = dg[k];
                    }
                    // the previous tile's MMAs over this part are done
                    if (h == 0 && !first && !(part ? wait(kYFull, pyf) : wait(kReFree, prf))) {
                        ok = false;
                        break;
                    }
                    const uint32_t off = sw128_chunk(r, part * 4 + qq);
#pragma unroll
                    for (int k = 0; k < D; ++k)
                        *reinterpret_cast<uint4*>(sA + k * kSliceA + off) = make_uint4(w[k][0], w[k][1], w[k][2], w[k][3]);
                    if (part == 0 && qq == 0) {
                        // the row scale, for the recombination of this tile
                        // (the slot's previous tile was read before set X
                        // was released for the previous tile's MMAs)
                        s_eterm[it & 1][r] = eterm_of((int)em);
                        mbar_arrive(&bars[(it & 1) ? kEt1 : kEt0]);
                    }
                    if (h == 1) {
                        asm volatile("fence.proxy.async.shared::cta;");
                        mbar_arrive(&bars[part ? kImReady : kReReady]);
                    }
                }
                if (!ok) break;
            }
            first = false;
        }
    } else {
        // ---------------------------------------------------- recombination
        // thread <-> (row r = TMEM lane, complex columns [8 eh, 8 eh + 8) of
        // each half); set column m < 16 is the real part of complex column
        // 16 hh + m, m >= 16 the imaginary part of 16 hh + m - 16
        const int eh = warp >> 2;
        const int r = ((warp & 3) << 5) | lane;
        const uint64_t rowoff = row_off(r);
        const uint32_t lane_base = tmem + ((uint32_t)((warp & 3) * 32) << 16);
        // the accumulators of 4 complex columns m0 .. m0 + 3 of set hh as
        // the integers Y (re, im interleaved)
        auto load_y = [&](uint32_t set, int m0, long long y[8], Bar release) {
            if constexpr (D == 7) {
                // real parts, then imaginary parts: half the live accumulator
                // registers of loading both at once (eight accumulators)
#pragma unroll
                for (int part = 0; part < 2; ++part) {
                    uint32_t cc[kAcc][4];
#pragma unroll
                    for (int k = 0; k < kAcc; ++k) {
                        const uint32_t ta = set + (uint32_t)(k * kNH + m0 + 16 * part);
                        asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
                                     : "=r"(cc[k][0]), "=r"(cc[k][1]), "=r"(cc[k][2]), "=r"(cc[k][3])
                                     : "r"(ta));
                    }
                    asm volatile("tcgen05.wait::ld.sync.aligned;");
                    if (part == 1 && release != kBars) {
                        asm volatile("tcgen05.fence::before_thread_sync;");
                        mbar_arrive(&bars[release]);
                    }
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        uint32_t c1[kAcc];
#pragma unroll
                        for (int k = 0; k < kAcc; ++k) c1[k] = cc[k][u];
                        y[2 * u + part] = combine_y<D>(c1);
                    }
                }
                return;
            }
            uint32_t re[kAcc][4], im[kAcc][4];
#pragma unroll
            for (int k = 0; k < kAcc; ++k) {
                const uint32_t ta = set + (uint32_t)(k * kNH + m0);
                asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
                             : "=r"(re[k][0]), "=r"(re[k][1]), "=r"(re[k][2]), "=r"(re[k][3])
                             : "r"(ta));
                asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
                             : "=r"(im[k][0]), "=r"(im[k][1]), "=r"(im[k][2]), "=r"(im[k][3])
                             : "r"(ta + 16u));
            }
            asm volatile("tcgen05.wait::ld.sync.aligned;");
            if (release != kBars) {
                // the set's accumulators are all in registers: it may be refilled
                asm volatile("tcgen05.fence::before_thread_sync;");
                mbar_arrive(&bars[release]);
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                uint32_t cr[kAcc], ci[kAcc];
#pragma unroll
                for (int k = 0; k < kAcc; ++k) {
                    cr[k] = re[k][u];
                    ci[k] = im[k][u];
                }
                y[2 * u] = combine_y<D>(cr);
                y[2 * u + 1] = combine_y<D>(ci);
            }
        };
        auto store = [&](char* gb, int c0, const long long y[8], int eterm) {
            // whole 32-byte sectors where neighbouring columns share one
#pragma unroll
            for (int u = 0; u < 4; u += 2) {
                const int c = c0 + u;
                const double re0 = finish_y(y[2 * u], eterm + sF20[c]), im0 = finish_y(y[2 * u + 1], eterm + sF20[32 + c]);
                const double re1 = finish_y(y[2 * u + 2], eterm + sF20[c + 1]);
                const double im1 = finish_y(y[2 * u + 3], eterm + sF20[32 + c + 1]);
                if constexpr (PAIR) {
                    asm volatile("st.global.v4.f64 [%0], {%1, %2, %3, %4};" ::"l"(gb + coloff[c]), "d"(re0), "d"(im0),
                                 "d"(re1), "d"(im1)
                                 : "memory");
                } else {
                    *reinterpret_cast<double2*>(gb + coloff[c]) = make_double2(re0, im0);
                    *reinterpret_cast<double2*>(gb + coloff[c + 1]) = make_double2(re1, im1);
                }
            }
        };
        uint32_t px = 0, py = 0;
        int it = 0;
        for (bool more = next_segment(true); more; more = next_segment(false))
        for (uint32_t t = seg_begin(); t < seg_end(); t += seg_step(), ++it) {
            char* gb = tile_ptr(t) + rowoff;
            const int slot = it & 1;
            uint32_t pet = (uint32_t)(it >> 1) & 1u;     // each slot completes every other tile
            if (!wait(slot ? kEt1 : kEt0, pet)) break;
            const int eterm = s_eterm[slot][r];
            bool ok = true;
#pragma unroll 1
            for (int hh = 0; hh < 2; ++hh) {
                if (!wait(hh ? kYFull : kXFull, hh ? py : px)) {
                    ok = false;
                    break;
                }
                asm volatile("tcgen05.fence::after_thread_sync;");
                const uint32_t set = lane_base + (hh ? kSetY : 0u);
                long long ya[8], yb[8];
                load_y(set, 8 * eh, ya, kBars);
                load_y(set, 8 * eh + 4, yb, hh ? kYFree : kXFree);
                store(gb, 16 * hh + 8 * eh, ya, eterm);
                store(gb, 16 * hh + 8 * eh + 4, yb, eterm);
            }
            if (!ok) break;
            if (kDft && eterm == kEtermBad) {   // an infinity or NaN among the row's inputs
                const double nan = __hiloint2double(0x7FF80000, 0);
#pragma unroll 1
                for (int c = 8 * eh; c < 32; c = (c & 7) == 7 ? c + 9 : c + 1)
                    *reinterpret_cast<double2*>(gb + coloff[c]) = make_double2(nan, nan);
            }
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    if (warp == kMmaWarp) {
        asm volatile("tcgen05.fence::after_thread_sync;");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols));
    }
}

template <int D>
void launch_impl(qe_state* s, const int* qubits, const cd* U, const char* tag) {
    if (s->dtype != QE_C128) fail(QE_ERR_UNSUPPORTED, "this tensor-core path is for complex128 states");
    if (s->n < 12) fail(QE_ERR_UNSUPPORTED, "tensor-core gates need n >= 12");
    const tc::Geometry g = tc::tile_geometry(qubits);
    GateArgs arg{};
    OzArgs& a = arg.z;
    a.x = reinterpret_cast<double2*>(s->d);
    a.L = g.L;
    a.kh = g.kh;
    std::memcpy(a.hq, g.hq, sizeof(g.hq));
    std::memcpy(a.gpos, g.gpos, sizeof(a.gpos));
    a.ntiles = 1ull << (s->n - 12);
    // the copy is ordered after the previous block on the stream and returns
    // once U is staged: no wait between blocks, and nothing to split on the host
    static_assert(sizeof(cd) == sizeof(double2), "interleaved complex");
    double2* const dU = reinterpret_cast<double2*>(ensure_scratch(s, 32 * 32 * sizeof(double2)));
    QE_CUDA(cudaMemcpyAsync(dU, U, 32 * 32 * sizeof(double2), cudaMemcpyHostToDevice, s->stream));
    arg.U = dU;
    a.status = status_word(s);
    a.spin_limit = 1ll << 21;   // polls of up to kSuspendNs each
    // Failure-path test (QE_TEST_STALL_TC128=1): the load warps withhold the
    // arrival for the first staged half, so the splitters' wait runs out after
    // a short limit, every role leaves through the shared abort flag, and the
    // host reports QE_ERR_TIMEOUT with the context intact.
    const char* stall = std::getenv("QE_TEST_STALL_TC128");
    a.stall_test = (stall != nullptr && stall[0] == '1') ? 1 : 0;
    if (a.stall_test) a.spin_limit = 1ll << 12;
    const size_t smem = oz_smem<D>();
    auto fn = qubits[0] == 0 ? k_gate_tc5_c128<D, true, GateArgs> : k_gate_tc5_c128<D, false, GateArgs>;
    QE_CUDA(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    const uint64_t grid = std::min<uint64_t>(a.ntiles, (uint64_t)num_sms());
    Launch Lc(s, tag, 2.0 * dim(s) * amp_bytes(s));
    fn<<<(unsigned)grid, kOzThreads, smem, s->stream>>>(arg);
    QE_CUDA(cudaGetLastError());
}

}  // namespace

// Apply a 5-qubit block to a complex128 state with the tensor cores: 56-bit
// splitting (seven digits) in the FP64 mode, 48-bit (six) in the fast
// double-float mode.
void launch_gate_tc5_c128(qe_state* s, const int* qubits, const cd* U) {
    if (s->arith == QE_ARITH_DF64) launch_impl<6>(s, qubits, U, "gate_tc_k5_c128_df");
    else launch_impl<7>(s, qubits, U, "gate_tc_k5_c128");
}

// One digit of a Fourier transform on a complex128 state (n >= 12): the qubits
// [q0, q0 + d), 1 <= d <= 5, whose matrix depends on the P qubits above them
// (P + d <= 20, n - 12 - P >= 0), of a register from qubit lo on.  With d < 5 the
// block is filled up with qubits of the register below the digit, so that its
// 32 amplitudes, which share a scale, stay within the register: with those that
// the tile has anyway if there are such (17 qubits from 5 on at n = 27 5.84 ms,
// 5.96 with the ones next to the digit), and not with qubit 0, whose blocks are
// the slower ones.  A register of fewer than five qubits takes in others.  `roots` holds the 2^(P + d) roots of unity
// of the transform's sign; `reversed`: leave the output bit-reversed.  56-bit
// splitting in both arithmetic modes (the seventh digit costs 3 %).
void launch_dft_digit_c128(qe_state* s, int lo, int q0, int d, int P, bool reversed, const double2* roots) {
    constexpr int D = 7;
    if (d < 1 || d > 5 || s->n < 12 + P) fail(QE_ERR_UNSUPPORTED, "transform digits need 1 to 5 qubits and n >= 12 + P");
    static thread_local DftArgs f;
    std::memset(&f, 0, sizeof(f));
    OzArgs& a = f.z;
    a.x = reinterpret_cast<double2*>(s->d);
    a.ntiles = 1ull << (s->n - 12);
    f.P = P;
    f.vlo = q0 + d;
    f.d = d;
    f.reversed = reversed;
    f.scale = std::pow(2.0, -0.5 * d);
    f.roots = roots;
    f.lt = s->n - 12 - P;
    // The block: the digit and, for d < 5, idle qubits; the tile: the block and
    // the lowest qubits outside it and the matrix bits.
    bool matrix[64] = {}, local[64] = {};
    for (int j = 0; j < P; ++j) matrix[f.vlo + j] = true;
    int gate[5], ng = 0;
    auto take = [&](int q) {
        gate[ng++] = q;
        local[q] = true;
        f.below += q < q0;
    };
    for (int j = 0; j < d; ++j) take(q0 + j);
    for (int q = std::min(q0 - 1, 11 - d); q >= std::max(lo, 1) && ng < 5; --q) take(q);
    for (int q = q0 - 1; q >= std::max(lo, 1) && ng < 5; --q)
        if (!local[q]) take(q);
    for (int q = q0 + d; q < 12 && ng < 5; ++q)
        if (!matrix[q]) take(q);
    for (int q = std::min(q0 - 1, 11 - d); q >= 0 && ng < 5; --q)
        if (!local[q]) take(q);
    for (int q = q0 + d; ng < 5; ++q)
        if (!matrix[q] && !local[q]) take(q);
    int nlocal = 5;
    for (int q = 0; nlocal < 12; ++q)
        if (!local[q] && !matrix[q]) {
            local[q] = true;
            ++nlocal;
        }
    std::sort(gate, gate + 5);
    const bool pair = gate[0] == 0;
    while (local[a.L]) ++a.L;
    if (a.L > 12) a.L = 12;
    if (a.L < 3) fail(QE_ERR_UNSUPPORTED, "transform digits need runs of eight amplitudes");
    int pos[64];
    for (int q = 0; q < s->n; ++q) {
        pos[q] = q < a.L ? q : a.L + a.kh;
        if (q >= a.L && local[q]) a.hq[a.kh++] = (uint8_t)q;
        if (q >= a.L && (local[q] || matrix[q])) f.skip[f.nskip++] = (uint8_t)q;
    }
    for (int j = 0; j < 5; ++j) a.gpos[j] = (uint8_t)pos[gate[j]];
    a.status = status_word(s);
    a.spin_limit = 1ll << 21;
    const size_t smem = oz_smem<D>();
    auto fn = pair ? k_gate_tc5_c128<D, true, DftArgs> : k_gate_tc5_c128<D, false, DftArgs>;
    QE_CUDA(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    const uint64_t grid = std::min<uint64_t>(a.ntiles, (uint64_t)num_sms());
    // The number of teams that makes the longest CTA's work the shortest: its
    // segments, each a share of the matrix's tiles and about 1.6 tiles' time to
    // drain, rebuild and refill the pipeline.
    double best = 1e300;
    for (int teams = 1; teams <= (int)std::min<uint64_t>(grid, 1ull << P); ++teams) {
        const double segs = std::ceil((double)(1ull << P) / teams);
        const double time = segs * (std::ceil((double)(1ull << f.lt) / (double)(grid / teams)) + 1.6);
        if (time < best) {
            best = time;
            f.teams = teams;
        }
    }
    Launch Lc(s, "gate_tc_k5_c128", 2.0 * dim(s) * amp_bytes(s));
    fn<<<(unsigned)grid, kOzThreads, smem, s->stream>>>(f);
    QE_CUDA(cudaGetLastError());
}

}  // namespace qe
