// Split-precision expansion (Eq. 7) on the 5th-generation tensor cores.
//
//   out[(j,j'), (n,n')] = sum_k P[(j,j')][k] * A[(n,n')][k]
//
// Both FP64 operands are split row by row into S bf16 slices (an error-free
// splitting in the manner of Ozaki, Ogita, Oishi & Rump 2012): with 2^e the
// smallest power of two above the row's largest magnitude, x 2^(8+9(S-1)-e) is
// rounded to an integer whose balanced base-512 digits d_0 .. d_{S-1} (|d_i| <=
// 256, which bf16 holds exactly) are the slices, d_i 2^(-8-9i) apart from 2^e.
// Products of slice i of a panel row with slice l of a coefficient row are
// integer multiples of 2^(-16-9s), s = i + l; those with i + l < S are formed,
// and summed per s by tcgen05.mma (kind::f16, FP32 accumulation in tensor
// memory).  Up to 256 / (s + 1) terms every partial sum of such a sum stays
// within 2^24 units, so the FP32 accumulation is exact; then the epilogue
// takes the accumulator out and it starts again from zero.
//
// Mixed build: S = 5 (44 bits, 15 products).  s = 0, 1, 2 have accumulators of
// their own, drained every 256, 128 and 64 terms into a double-float sum; s = 3
// and 4 share the fourth, which need not be exact (its rounding is 2^-47 of
// the row scales per product) and is added every 512 terms.  With base-128 digits the
// same accuracy took 6 slices and 21 products, and all pairs s >= 3 shared an
// accumulator seven bits further up: the sums here are 6 to 9 times closer to
// 64 bits (4.5e-12 -> 7e-13 at 2422 labels, 1.7e-12 -> 1.8e-13 at 1367).  2422
// labels x 1275 columns x 160000 rows: 14.2 -> 10.4 ms (8.8 with f32x2 sums), 1367 x 210 x 22500: 358
// -> 266 us.
//
// FP64 build: S = 7 (62 bits, 28 products), every s with an accumulator of its
// own, and the row exponents kept apart from the digits.  The drained sums are
// integers and are added as such (two 64-bit words per element, s <= 2 and
// s >= 3), so the element is the correctly rounded sum of the products of the
// operands' 62 leading bits, whatever the order of the labels.  The FP64 pipe of
// this part runs at a 1/1000 of the tensor rate: its sums took 14.0 ms where this
// takes 0.65 ms (12.9 GFLOP), and rounded every one of the 1367 additions.
//   What the digits leave out is relative to the largest entries of the two rows:
// K labels err by less than K 2^-60 of their product, typically by 2^-63 sqrt(K),
// and sums in FP64 by about 2^-54 M, M = sum |p_k a_k|.  Where the large entries of
// the one row meet zeros or tiny entries of the other (h_jj' of 50 and S = 0
// between groups, beside integrals of 1e-6) M can be so small that FP64 is closer.
// So the FP64 build carries an eighth slice, the magnitudes to 8 bits rounded down,
// whose product is a lower bound of M: an element with 0 < M < sqrt(K') 2^-9 of the
// scales (K' nonzero entries in the row that has fewer; there the typical errors are
// alike; at least 2^-7, where the bounds are)
// is summed in FP64 (fp64_elements_kernel).  Magnitudes below 2^-9 count as 2^-40,
// so M = 0 means that no two entries meet, and the sum is exactly zero; a row with a
// value that is not finite is all 2^-40.  Molecular integrals with dense target
// densities lie above the line (the lowest 1e-3 of M at 0.05 to 0.6 of the scales, the
// line at 0.01 to 0.08); densities of a few entries, between small groups of a batch
// over symmetries, leave 0.1 % of the elements below it.
// The magnitudes are multiplied by a launch of their own (this kernel with one
// slice and 128-wide tiles), which leaves a bit an element, beside what comes before
// the digits: an eighth pair of tiles in every stage of those made them 22 % slower
// (0.65 -> 0.79 ms).
//
// Kernel structure (persistent CTAs on 128 x TBN output tiles, 10 warps):
//   warp 0  TMA producer: per K stage (32 or 64 labels) and slice, one panel
//           tile and one coefficient tile into a slot of a ring of as many
//           slots as fit, with full/empty mbarriers
//   warp 1  MMA issuer (one elected thread), TMEM allocation owner
//   warps 2-9 epilogue: TMEM -> registers, accumulation, FP64 out (two warps
//           per TMEM lane quadrant)
// A stage takes the pairs of the inexact accumulator first, those with slice 0
// last, and then s = S-1 .. 0 of the exact ones.  So an accumulator due for draining is drained
// behind the pairs that follow and those of the next stage that precede its
// own (each accumulator has its own full/empty barriers), and slices S-1 .. 0
// are released in that order, which is the order of the ring.
// Every mbarrier wait is bounded; on a timeout the kernel records an error,
// drains its own copies and MMAs, frees TMEM and returns.
//
// Rows with j == j' carry h_jj and the delta_jj' E term and so have a wide
// dynamic range; the kernel skips them and diag_rows_kernel computes them (in
// double-float or FP64).
#include <cuda.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <mutex>

#include "hb_api_internal.cuh"
#include "hb_plan.cuh"
#include "hb_split.cuh"
#include "hb_df.cuh"
#include "hb_tc.cuh"

namespace hb {

// Panel slices of one precision, and their tensor maps.
struct PanelSlices {
    int slices = 0;
    __nv_bfloat16 *buf = nullptr;            // [S][Kpad/64][n_co*n_co][64] (FP64: S + 1, the last the magnitudes)
    RowScale *scales = nullptr;              // FP64: those of the rows [n_co*n_co]
    // [stage width 32, 64][box of 8 x 16, 16 x 8, 32 x 4 continuum pairs (j' x j)]
    CUtensorMap tm[2][3];
    bool ready = false, borrowed = false;
};

struct MixedState {
    PanelSlices panel[2];                    // HB_FP64, HB_MIXED
    float2 *pdiag = nullptr;                 // mixed: diagonal panel rows (j, j) as float pairs [n_co][Kpad]
};

}  // namespace hb

using namespace hb;

namespace {

using namespace hb::tc;

constexpr int BM = 128, BN = 128, BKB = 64;  // tile rows, tile cols, K per block (one 128-B swizzle row)
constexpr int KCHUNK = 512;                  // exact FP32 accumulation span
constexpr int MAXS = 6;
constexpr int A_TILE = BM * BKB * 2;         // 16 KB
constexpr int B_TILE = BN * BKB * 2;         // 16 KB
constexpr int SLOT = A_TILE + B_TILE;        // one slice of one K block (S slots in shared memory)
constexpr int TMEM_COLS = 512;               // 4 accumulators x 128 columns
constexpr int EPI_WARPS = 8;                 // 2 per TMEM lane quadrant
constexpr int EPI_THREADS = 32 * EPI_WARPS;
constexpr int EPI_COLS = BN / 2;             // columns per epilogue thread
constexpr int NTHREADS = 64 + EPI_THREADS;

// The expansion kernel's K pipeline: stages of KS = 32 labels (64-byte operand
// rows, 64-byte swizzle) or 64 (128-byte rows and swizzle), and a ring of as
// many slice slots as fit, so the copies of the next stages are in flight
// while the stages before them are multiplied.  Its tile is 128 continuum
// pairs x TBN columns (state pairs), TBN = 32, 64 or 128 chosen per merged
// block from its column count.  64-K stages serve 128-column tiles over long K
// (fewer waits and copies per K), 32-K stages the rest (deeper prefetch).
constexpr int XBUDGET = 7 * 32 * 1024;       // shared memory of the slots
constexpr int XBARS = 24;                    // full and empty barriers: slots at most
constexpr int XACC = 7;                      // accumulators at most
constexpr int kK64Blocks = 32;               // 64-K stages from this many 64-wide K blocks up
constexpr int kF64Slices = 7;                // digit slices of the FP64 build
constexpr int kF64Planes = kF64Slices + 1;   // and its magnitudes
constexpr int kWeakSlots = 3;                // ring of the magnitudes' launch, whose CTAs fit beside class 4's
// what the kernel computes: the mixed and the FP64 build's sums, and the bits of
// the elements whose magnitudes are too small for the digits
enum : int { kMixedSums, kF64Sums, kWeakBits };
__host__ __device__ constexpr int xa_tile(int ks) { return BM * ks * 2; }
// one slice of one stage: panel tile, then coefficient tile (multiples of 1 KB)
__host__ __device__ constexpr int xslot(int tbn, int ks) { return (BM + tbn) * ks * 2; }
__host__ __device__ constexpr int xslots(int tbn, int ks) {
    return XBUDGET / xslot(tbn, ks) < XBARS ? XBUDGET / xslot(tbn, ks) : XBARS;
}
// accumulators: one per s below NEX, one for the rest
__host__ __device__ constexpr int xaccs(int S, int nex) { return S <= nex ? S : nex + 1; }
__host__ __device__ constexpr int xtmem_cols(int accs, int tbn) {
    int c = 32;
    while (c < accs * tbn) c *= 2;
    return c;
}
// stages between drains of accumulator a: 256 / (a + 1) labels, rounded down to
// a power of two, for an exact one, 512 for the inexact one
__host__ __device__ constexpr int xperiod(int a, int nex, int ks) {
    return (a >= nex ? 512 : a == 0 ? 256 : a == 1 ? 128 : a <= 3 ? 64 : 32) / ks;
}
// Whether accumulator a is drained after stage ks of nst.  a = 0 is drained
// between the stages at which a = 1 is, so that at most two of the first three
// come at once.  Without exact accumulators (magnitudes) the end alone counts.
template <int NEX, int KS>
__device__ __forceinline__ bool acc_due(int a, int ks, int nst) {
    if (NEX == 0) return ks == nst - 1;
    const int per = xperiod(a, NEX, KS);
    return ks == nst - 1 || (ks + 1 + (a == 0 ? per / 4 : 0)) % per == 0;
}

// The pairs (i, l) of a stage in order.
struct PairOrder {
    int n = 0;
    int i[28] = {}, l[28] = {};
};
template <int S, int NEX>
__host__ __device__ constexpr PairOrder pair_order() {
    PairOrder o;
    for (int m = S - 1; m >= 0; --m)              // inexact pairs, by their lower slice
        for (int s = S - 1; s >= NEX; --s)
            for (int i = 0; i <= s; ++i)
                if ((i < s - i ? i : s - i) == m) {
                    o.i[o.n] = i;
                    o.l[o.n++] = s - i;
                }
    for (int s = (S < NEX ? S : NEX) - 1; s >= 0; --s)
        for (int i = 0; i <= s; ++i) {
            o.i[o.n] = i;
            o.l[o.n++] = s - i;
        }
    return o;
}
// first and last pair that reads slice t; last pair of accumulator a
__host__ __device__ constexpr int first_use(const PairOrder &o, int t) {
    for (int p = 0; p < o.n; ++p)
        if (o.i[p] == t || o.l[p] == t) return p;
    return -1;
}
__host__ __device__ constexpr int last_use(const PairOrder &o, int t) {
    int r = -1;
    for (int p = 0; p < o.n; ++p)
        if (o.i[p] == t || o.l[p] == t) r = p;
    return r;
}
__host__ __device__ constexpr int last_of_acc(const PairOrder &o, int a, int nex) {
    int r = -1;
    for (int p = 0; p < o.n; ++p) {
        const int s = o.i[p] + o.l[p];
        if ((s < nex ? s : nex) == a) r = p;
    }
    return r;
}
__host__ __device__ constexpr int first_of_acc(const PairOrder &o, int a, int nex) {
    for (int p = 0; p < o.n; ++p) {
        const int s = o.i[p] + o.l[p];
        if ((s < nex ? s : nex) == a) return p;
    }
    return -1;
}

__device__ __forceinline__ void tma_load_4d(void *dst, const CUtensorMap *tm, uint64_t *bar, int c0, int c1, int c2,
                                            int c3) {
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6}], "
        "[%2];" ::"r"(smem_u32(dst)),
        "l"((uint64_t)tm), "r"(smem_u32(bar)), "r"(c0), "r"(c1), "r"(c2), "r"(c3)
        : "memory");
}

__device__ __forceinline__ void tma_load_3d(void *dst, const CUtensorMap *tm, uint64_t *bar, int c0, int c1,
                                            int c2) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], "
        "[%2];" ::"r"(smem_u32(dst)),
        "l"((uint64_t)tm), "r"(smem_u32(bar)), "r"(c0), "r"(c1), "r"(c2)
        : "memory");
}

// Slot of slice t in a K block of parity P.  Slice i of a block is last read
// at step max(i, S-1-i) (steps follow the slices as they arrive), so in odd
// blocks the first-needed slices go to the slots that the even block frees
// first, and the loads of a block overlap the last steps of the one before.
template <int S>
__host__ __device__ constexpr int release_step(int i) { return i > S - 1 - i ? i : S - 1 - i; }

template <int S>
__host__ __device__ constexpr int slot_of(int P, int t) {
    if (P == 0) return t;
    // the slot whose release rank (release step, then index) is t
    for (int i = 0; i < S; ++i) {
        int r = 0;
        for (int j = 0; j < S; ++j)
            r += (release_step<S>(j) < release_step<S>(i)) || (release_step<S>(j) == release_step<S>(i) && j < i);
        if (r == t) return i;
    }
    return 0;
}

// One K block of MMAs, fully unrolled for slot parity P: for each arriving
// slice t, the pairs (i, l) with max(i, l) = t and i + l < S, then the commits
// that free the slots read for the last time.
template <int S, int P>
__device__ __forceinline__ bool mma_block(uint64_t *full_bar, uint64_t *empty_bar, uint32_t par, uint32_t tmem,
                                          uint64_t desc0, uint32_t idesc, uint32_t &fresh, int *err) {
#pragma unroll
    for (int t = 0; t < S; ++t) {
        if (!mbar_wait(&full_bar[slot_of<S>(P, t)], par, err, 4)) return false;
        tc_fence_after();
#pragma unroll
        for (int i = 0; i <= t; ++i) {
#pragma unroll
            for (int l = 0; l <= t; ++l) {
                if ((i == t || l == t) && i + l < S) {
                    const int s = i + l < 3 ? i + l : 3;
                    const uint32_t offA = (uint32_t)(slot_of<S>(P, i) * SLOT);
                    const uint32_t offB = (uint32_t)(slot_of<S>(P, l) * SLOT + A_TILE);
#pragma unroll
                    for (int k = 0; k < BKB / 16; ++k) {
                        const uint32_t acc = (fresh >> s) & 1u ? 0u : 1u;
                        mma_bf16(tmem + s * BN, desc0 + ((offA + k * 32) >> 4), desc0 + ((offB + k * 32) >> 4), idesc,
                                 acc);
                        fresh &= ~(1u << s);
                    }
                }
            }
        }
#pragma unroll
        for (int i = 0; i < S; ++i)
            if (release_step<S>(i) == t) mma_commit(&empty_bar[slot_of<S>(P, i)]);
    }
    return true;
}

// What the MMA issuer carries through a launch.  due: the accumulators drained
// after the current stage; fresh: those whose next MMA starts from zero; used:
// those handed over before; epar: the parity of each one's next hand-back.
struct MmaState {
    uint64_t *full_bar, *empty_bar, *acc_full, *acc_empty;
    uint32_t tmem, idesc;
    uint64_t desc0;
    int *err;
    uint32_t due = 0, fresh = 0, used = 0, epar = 0;
    uint32_t leader = 0;      // this lane issues
};

// Pair P of a stage and those after it; slice t of the stage is in slot sl[t],
// whose use has parity sp[t].
template <int S, int NEX, int TBN, int KS, int P>
__device__ __forceinline__ bool mma_pairs(MmaState &m, const int (&sl)[S], const uint32_t (&sp)[S]) {
    constexpr PairOrder O = pair_order<S, NEX>();
    constexpr int XS = xslot(TBN, KS);
    constexpr int i = O.i[P], l = O.l[P], a = i + l < NEX ? i + l : NEX;
    constexpr bool wait_i = first_use(O, i) == P, wait_l = l != i && first_use(O, l) == P;
    constexpr bool first_a = first_of_acc(O, a, NEX) == P, last_a = last_of_acc(O, a, NEX) == P;
    if (wait_i && !mbar_wait_warp(&m.full_bar[sl[i]], sp[i], m.err, 4)) return false;
    if (wait_l && !mbar_wait_warp(&m.full_bar[sl[l]], sp[l], m.err, 4)) return false;
    if (first_a && (m.fresh >> a) & 1u) {
        // the epilogue has taken this accumulator's last sums
        if ((m.used >> a) & 1u) {
            if (!mbar_wait_warp(&m.acc_empty[a], (m.epar >> a) & 1u, m.err, 3)) return false;
            m.epar ^= 1u << a;
        }
        m.used |= 1u << a;
    }
    if (wait_i || wait_l || first_a) tc_fence_after();
    const uint64_t da = m.desc0 + (uint32_t)((sl[i] * XS) >> 4), db = m.desc0 + (uint32_t)((sl[l] * XS + xa_tile(KS)) >> 4);
#pragma unroll
    for (int k = 0; k < KS / 16; ++k) {
        const uint32_t acc = (first_a && k == 0) ? (~(m.fresh >> a) & 1u) : 1u;
        mma_bf16_elect(m.tmem + a * TBN, da + 2 * k, db + 2 * k, m.idesc, acc, m.leader);
    }
    if (first_a) m.fresh &= ~(1u << a);
    if (last_use(O, i) == P) mma_commit_elect(&m.empty_bar[sl[i]], m.leader);
    if (l != i && last_use(O, l) == P) mma_commit_elect(&m.empty_bar[sl[l]], m.leader);
    if (last_a && (m.due >> a) & 1u) {
        mma_commit_elect(&m.acc_full[a], m.leader);
        m.fresh |= 1u << a;
    }
    if constexpr (P + 1 < O.n) return mma_pairs<S, NEX, TBN, KS, P + 1>(m, sl, sp);
    return true;
}

// One K stage of the expansion kernel.  Its slices lie in the ring from slot
// `slot0` on, slice S-1 first, `par` being the parity of that slot's use
// (flipped where the ring wraps).
template <int S, int NEX, int TBN, int KS, int NS>
__device__ __forceinline__ bool mma_stage(MmaState &m, int slot0, uint32_t par) {
    int sl[S];
    uint32_t sp[S];
#pragma unroll
    for (int t = 0; t < S; ++t) {
        const int x = slot0 + (S - 1 - t);
        sl[t] = x >= NS ? x - NS : x;
        sp[t] = x >= NS ? par ^ 1u : par;
    }
    return mma_pairs<S, NEX, TBN, KS, 0>(m, sl, sp);
}

// One drained accumulator of the mixed kernel (NC columns of this thread's
// TMEM lane): an exact one by TwoSum (2^-18 of the result for s = 2 still needs
// it to keep the low word below an ulp of the high one), the inexact one
// (2^-27) into the low word.
template <bool EXACT, int NP>
__device__ __forceinline__ void drain_df(uint32_t taddr, f2 (&hi)[NP], f2 (&lo)[NP]) {
    constexpr int NC = 2 * NP;
    static_assert(NC % 16 == 0, "columns are loaded 16 at a time");
#pragma unroll
    for (int c0 = 0; c0 < NC; c0 += 32) {
        uint32_t v[16], w[16];
        tmem_ld16_async(taddr + c0, v);
        if (c0 + 16 < NC) tmem_ld16_async(taddr + c0 + 16, w);
        tmem_wait_ld();
        tmem_regs_ready(v);
        if (c0 + 16 < NC) tmem_regs_ready(w);
        fold16<EXACT>(v, &hi[c0 / 2], &lo[c0 / 2]);
        if (c0 + 16 < NC) fold16<EXACT>(w, &hi[(c0 + 16) % NC / 2], &lo[(c0 + 16) % NC / 2]);
    }
}

// One drained accumulator of the FP64 kernel: its sums are integers of
// 2^(-16-9s), added to word 0 (units of 2^-34, s <= 2) or 1 (2^-70).
template <int SS, int NC>
__device__ __forceinline__ void drain_int(uint32_t taddr, long long (&acc)[2][NC]) {
    static_assert(NC % 16 == 0, "columns are loaded 16 at a time");
    constexpr int w = SS <= 2 ? 0 : 1;
    constexpr float to_int = (float)(1ull << (SS <= 2 ? 16 + 9 * SS : 0)) * 1.0f;
    constexpr int lift = SS <= 2 ? 9 * (2 - SS) : 9 * (6 - SS);
#pragma unroll
    for (int c0 = 0; c0 < NC; c0 += 16) {
        uint32_t v[16];
        tmem_ld16_async(taddr + c0, v);
        tmem_wait_ld();
        tmem_regs_ready(v);
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            float x = __uint_as_float(v[i]);
            if constexpr (SS <= 2) x *= to_int;
            else x = x * (float)(1ull << 40) * (float)(1ull << (16 + 9 * SS - 40));
            acc[w][c0 + i] += (long long)__float2int_rn(x) * (1ll << lift);
        }
    }
}

// The magnitude sums of 32 columns, of which n exist: bit c set where the digits of
// column c are not good enough (see the head of this file).
__device__ __forceinline__ uint32_t drain_weak(uint32_t taddr, float line, const RowScale *__restrict__ cols, int n) {
    uint32_t weak = 0;
#pragma unroll
    for (int c0 = 0; c0 < 32; c0 += 16) {
        uint32_t v[16];
        tmem_ld16_async(taddr + c0, v);
        tmem_wait_ld();
        tmem_regs_ready(v);
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            const float x = __uint_as_float(v[i]);
            if (c0 + i < n && x > 0.0f && x < fminf(line, __ldg(&cols[c0 + i].line))) weak |= 1u << (c0 + i);
        }
    }
    return weak;
}

// The FP64 element of the two words and the row and column exponents.
constexpr int kExpNaN = 1 << 20;               // exponent of a row with a value that is not finite
__device__ __forceinline__ double int_words_to_double(long long a, long long b, int ea, int eb) {
    if (ea == kExpNaN || eb == kExpNaN) return __longlong_as_double(0x7FF8000000000000ll);
    const double v = fma((double)b, 0x1p-36, (double)a);
    const int e = ea + eb - 34;
    // |v| < 2^53: a power of two in the normal range leaves v in it, or takes it below
    if (e > -960 && e < 960) return v * __hiloint2double((e + 1023) << 20, 0);
    return scalbn(v, e);
}

// Fold one chunk's accumulators (NC columns of this thread's TMEM lane,
// accumulator s at column offset s * stride) into the double-float sums:
// s = 0, 1, 2 by TwoSum (2^-14 of the result for s = 2 still needs it to keep
// the low word below an ulp of the high one), s >= 3 (2^-21) into the low word.
template <int S, int NP>
__device__ __forceinline__ void drain_chunk(uint32_t tbase, int stride, f2 (&hi)[NP], f2 (&lo)[NP]) {
    constexpr int NC = 2 * NP;
    constexpr int n_acc = S < 4 ? S : 4;       // accumulators written by the MMAs
    static_assert(NC % 16 == 0, "columns are loaded 16 at a time");
#pragma unroll
    for (int c0 = 0; c0 < NC; c0 += 16) {
        // two accumulators' 16 columns in flight together, one wait each pair
        uint32_t v[16], w[16];
        tmem_ld16_async(tbase + c0, v);
        if (n_acc > 1) tmem_ld16_async(tbase + stride + c0, w);
        tmem_wait_ld();
        tmem_regs_ready(v);
        fold16<true>(v, &hi[c0 / 2], &lo[c0 / 2]);
        if (n_acc > 1) {
            tmem_regs_ready(w);
            fold16<true>(w, &hi[c0 / 2], &lo[c0 / 2]);
        }
        if (n_acc > 2) {
            tmem_ld16_async(tbase + 2 * stride + c0, v);
            if (n_acc > 3) tmem_ld16_async(tbase + 3 * stride + c0, w);
            tmem_wait_ld();
            tmem_regs_ready(v);
            fold16<true>(v, &hi[c0 / 2], &lo[c0 / 2]);
            if (n_acc > 3) {
                tmem_regs_ready(w);
                fold16<false>(w, &hi[c0 / 2], &lo[c0 / 2]);
            }
        }
    }
}

// Position of tile `tile` of a grouped launch: its task, the first rows of
// its continuum-pair block and its first column.
struct TilePos {
    int ti, jj0, jjp0, n0;
};

template <int TBN>
__device__ __forceinline__ TilePos tile_pos(const SplitTask *__restrict__ tasks, const int64_t *__restrict__ blk,
                                            int n_tasks, int tile) {
    TilePos p;
    p.ti = task_of(blk, n_tasks, tile);
    const int lb = (int)(tile - __ldg(blk + p.ti));
    const SplitTask &a = tasks[p.ti];
    const int ntn = a.ntn, jpt_tiles = a.jpt_tiles, lg = a.bjp_log2;
    const int tile_n = lb % ntn, tile_m = lb / ntn;   // N fastest: CTAs sharing a panel tile run together
    p.jj0 = (tile_m / jpt_tiles) * (BM >> lg);        // tile of (128 >> lg) j x (1 << lg) j'
    p.jjp0 = (tile_m % jpt_tiles) << lg;
    p.n0 = tile_n * TBN;
    return p;
}

// Persistent: each CTA takes tiles blockIdx.x, blockIdx.x + gridDim.x, ...
// The slot ring, the accumulator hand-over and their barrier phases run on
// across tiles, so the loads and MMAs of the next tile start while the
// epilogue warps still write the last one out from registers.  kF64Sums: the FP64
// build's kernel (integer sums, exponents apart: pscale of the panel's rows,
// n_co x n_co, cscale of the coefficient rows).  kWeakBits: a bit an element in `weak`,
// set where the sum of the magnitudes (plane `plane0` of the slices) is below the
// lines of its rows.
template <int S, int TBN, int KS, int MODE>
__global__ void __launch_bounds__(NTHREADS, 1)
split_expand_kernel(const __grid_constant__ CUtensorMap tm_panel, const __grid_constant__ CUtensorMap tm_coef,
                    const SplitTask *__restrict__ tasks, const int64_t *__restrict__ blk, int n_tasks, int n_tiles,
                    int kblocks, int coef_planes, const ExpCol *__restrict__ cols, const RowScale *__restrict__ pscale,
                    const RowScale *__restrict__ cscale, uint32_t *__restrict__ weak, int plane0, int n_co, int *err, int shard_r, int shard_n) {
    // this launch's tiles: shard_r, shard_r + shard_n, ... (all of them unless
    // sharded), numbered t = 0, 1, ... so that every role walks the same list
    const int n_local = n_tiles > shard_r ? (n_tiles - shard_r + shard_n - 1) / shard_n : 0;
    constexpr bool F64 = MODE == kF64Sums, WEAK = MODE == kWeakBits;
    constexpr int NEX = WEAK ? 0 : F64 ? S : 3;   // accumulators of one s each
    constexpr int NACC = xaccs(S, NEX);
    constexpr int XS = xslot(TBN, KS), NS = WEAK ? kWeakSlots : xslots(TBN, KS);
    constexpr int TCOLS = xtmem_cols(NACC, TBN);
    constexpr int ECOLS = TBN / 2;            // columns per epilogue thread
    static_assert(KS == 32 || KS == 64, "stage width");
    static_assert(NS >= S && NS <= XBARS && NACC <= XACC && TCOLS <= 512, "slots and tensor memory");
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    uint8_t *base = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint8_t *slots = base;                                         // [NS][XS]
    uint64_t *full_bar = (uint64_t *)(base + NS * XS);             // [XBARS]
    uint64_t *empty_bar = full_bar + XBARS;                        // [XBARS]
    uint64_t *acc_full = empty_bar + XBARS;                        // [XACC]
    uint64_t *acc_empty = acc_full + XACC;                         // [XACC]
    uint64_t *final_bar = acc_empty + XACC;                        // [1]
    uint32_t *tmem_slot = (uint32_t *)(final_bar + 1);
    // the epilogue's tile, double-buffered
    __shared__ SplitTask ta[2];
    __shared__ TilePos tp[2];
    __shared__ int epi_fail;                 // an epilogue wait gave up (read only after a barrier)

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int nst = kblocks * (64 / KS);     // K stages per tile

    if (threadIdx.x == 0) {
        epi_fail = 0;
        for (int i = 0; i < XBARS; ++i) { mbar_init(&full_bar[i], 1); mbar_init(&empty_bar[i], 1); }
        for (int b = 0; b < XACC; ++b) { mbar_init(&acc_full[b], 1); mbar_init(&acc_empty[b], EPI_THREADS); }
        mbar_init(final_bar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                     "r"(TCOLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    if (warp == 0) {
        // ------------------------------------------------------ TMA producer
        if (lane == 0) {
            int sl = 0, loads = 0;               // next slot, copies issued so far
            uint32_t par = 1;                    // parity of the release the slot waits for (none in the first round)
            bool ok = true;
            for (int t = blockIdx.x; t < n_local && ok; t += gridDim.x) {
                const int tile = shard_r + shard_n * t;
                const TilePos p = tile_pos<TBN>(tasks, blk, n_tasks, tile);
                const int cx = tasks[p.ti].cfp + p.jjp0, cy = tasks[p.ti].cf + p.jj0;
                const int crow = (int)(tasks[p.ti].coef_row0 + p.n0);
                const int kc0 = tasks[p.ti].kc0;      // the block's label class in the coefficient slices
                for (int ks = 0; ks < nst && ok; ++ks) {
                    const int kx = KS == 64 ? 0 : (ks & 1) * 32;   // part of 64-wide K block kb
                    const int kb = KS == 64 ? ks : ks >> 1;
                    for (int i = S - 1; i >= 0 && ok; --i) {
                        const int plane = i + (WEAK ? plane0 : 0);
                        if (loads >= NS) ok = mbar_wait(&empty_bar[sl], par, err, 1);
                        if (!ok) break;
                        uint8_t *sA = slots + sl * XS;
                        mbar_expect_tx(&full_bar[sl], (uint32_t)XS);
                        tma_load_4d(sA, &tm_panel, &full_bar[sl], kx, cx, cy, plane * kblocks + kb);
                        tma_load_3d(sA + xa_tile(KS), &tm_coef, &full_bar[sl], kx, crow,
                                    plane * coef_planes + kc0 + kb);
                        if (loads < 2 * NS) ++loads;
                        if (++sl == NS) { sl = 0; par ^= 1u; }
                    }
                }
            }
            // wait until this producer's last copy into every slot has landed
            // (slots before `sl` were last filled in this round, the others in the one before)
            for (int i = 0; i < NS && i < loads; ++i) {
                const uint32_t fp = i < sl ? par ^ 1u : par;
                mbar_wait(&full_bar[i], fp, err, 2);
            }
        }
    } else if (warp == 1) {
        // ------------------------------------------------------ MMA issuer
        MmaState m;
        m.full_bar = full_bar; m.empty_bar = empty_bar; m.acc_full = acc_full; m.acc_empty = acc_empty;
        m.tmem = __shfl_sync(0xffffffffu, tmem, 0);
        m.idesc = instr_desc_bf16(BM, TBN);
        // + (offset >> 4) per operand tile
        m.desc0 = KS == 64 ? smem_desc_sw128(smem_u32(slots)) : smem_desc_sw64(smem_u32(slots));
        m.err = err;
        m.fresh = (1u << NACC) - 1u;
        m.leader = elect_lane();
        bool ok = true;
        int sl = 0;
        uint32_t par = 0;
        for (int t = blockIdx.x; t < n_local && ok; t += gridDim.x)
            for (int ks = 0; ks < nst && ok; ++ks) {
                m.due = 0;
#pragma unroll
                for (int a = 0; a < NACC; ++a) m.due |= acc_due<NEX, KS>(a, ks, nst) ? 1u << a : 0u;
                ok = mma_stage<S, NEX, TBN, KS, NS>(m, sl, par);
                sl += S;
                if (sl >= NS) { sl -= NS; par ^= 1u; }
            }
        mma_commit_elect(final_bar, m.leader);
        mbar_wait_warp(final_bar, 0, err, 5);
    } else {
        // ------------------------------------------------------ epilogue
        const int e = threadIdx.x - 64;          // 0 .. EPI_THREADS-1
        const int ew = warp - 2;
        const int q = warp & 3;                  // TMEM lane quadrant this warp may access
        const int col0 = (ew >> 2) * ECOLS;
        const int row = q * 32 + lane;           // tile row = TMEM lane
        const uint32_t tq = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)col0;
        int it = 0;
        uint32_t fpar = 0;                       // parity of each accumulator's next hand-over
        for (int t = blockIdx.x; t < n_local; t += gridDim.x, ++it) {
            const int tile = shard_r + shard_n * t;
            const int buf = it & 1;
            // the buffer was last read by the stores of tile it-2, which every
            // epilogue warp finished before the barriers of tile it-1
            if (e == 0) {
                tp[buf] = tile_pos<TBN>(tasks, blk, n_tasks, tile);
                ta[buf] = tasks[tp[buf].ti];
            }
            // every epilogue thread reaches both barriers of a tile, so the
            // failure flag read after the first is the same for all of them
            named_bar_sync(1, EPI_THREADS);
            const bool failed = epi_fail != 0;
            named_bar_sync(1, EPI_THREADS);
            if (failed) break;
            const SplitTask &a = ta[buf];
            // the column records are read when the tile is written out
            if (e < TBN / 4 && tp[buf].n0 + 4 * e < a.N)
                asm volatile("prefetch.global.L1 [%0];" ::"l"(cols + a.col0 + tp[buf].n0 + 4 * e));
            f2 hi[MODE ? 1 : ECOLS / 2], lo[MODE ? 1 : ECOLS / 2];
            long long wd[2][F64 ? ECOLS : 1];
            uint32_t bits[2] = {0, 0};               // weak columns
            if constexpr (WEAK) {
            } else if constexpr (F64) {
#pragma unroll
                for (int c = 0; c < ECOLS; ++c) { wd[0][c] = 0; wd[1][c] = 0; }
            } else {
#pragma unroll
                for (int c = 0; c < ECOLS / 2; ++c) { hi[c] = f2_pack(0.0f, 0.0f); lo[c] = f2_pack(0.0f, 0.0f); }
            }
            bool ok = true;
            for (int ks = 0; ks < nst; ++ks) {
                // in the order in which the stage hands them over
#pragma unroll
                for (int b = NACC - 1; b >= 0; --b) {
                    if (!acc_due<NEX, KS>(b, ks, nst)) continue;
                    if (ok) ok = mbar_wait(&acc_full[b], (fpar >> b) & 1u, err, 6);
                    fpar ^= 1u << b;
                    if (!ok) continue;
                    tc_fence_after();
                    if constexpr (WEAK) {
                        const int jj = tp[buf].jj0 + (row >> a.bjp_log2), jjp = tp[buf].jjp0 + (row & ((1 << a.bjp_log2) - 1));
                        const float line = jj < a.cn && jjp < a.cnp
                                               ? __ldg(&pscale[(int64_t)(a.cf + jj) * n_co + a.cfp + jjp].line) : 0.0f;
                        const int n0 = tp[buf].n0 + col0;
#pragma unroll
                        for (int w = 0; w < 2; ++w)
                            bits[w] = drain_weak(tq + 32 * w, line, cscale + a.coef_row0 + n0 + 32 * w, a.N - n0 - 32 * w);
                    } else if constexpr (F64) {
                        if (b == 0) drain_int<0>(tq, wd);
                        else if (b == 1) drain_int<1>(tq + TBN, wd);
                        else if (b == 2) drain_int<2>(tq + 2 * TBN, wd);
                        else if (b == 3) drain_int<3>(tq + 3 * TBN, wd);
                        else if (b == 4) drain_int<4>(tq + 4 * TBN, wd);
                        else if (b == 5) drain_int<5>(tq + 5 * TBN, wd);
                        else drain_int<6>(tq + 6 * TBN, wd);
                    } else if (b < NEX) {
                        drain_df<true>(tq + b * TBN, hi, lo);
                    } else {
                        drain_df<false>(tq + b * TBN, hi, lo);
                    }
                    tc_fence_before();
                    mbar_arrive(&acc_empty[b]);
                }
            }
            if (!ok) {
                epi_fail = 1;
                continue;                        // leaves at the next tile's first barriers
            }
            // the accumulators are free again: the MMAs of the next tile run
            // while this one is written out
            const int lg = a.bjp_log2;
            const int jj = tp[buf].jj0 + (row >> lg), jjp = tp[buf].jjp0 + (row & ((1 << lg) - 1));
            const bool in = jj < a.cn && jjp < a.cnp && (a.cf + jj) != (a.cfp + jjp);
            if constexpr (WEAK) {
                const int w0 = (tp[buf].n0 + col0) >> 5;
#pragma unroll
                for (int w = 0; w < 2; ++w)
                    if (in && 32 * (w0 + w) < a.N)
                        weak[a.weak0 + (int64_t)(w0 + w) * a.cn * a.cnp + (int64_t)jj * a.cnp + jjp] = bits[w];
            } else if (in) {
                const int n0 = tp[buf].n0 + col0;
                const int4 *__restrict__ cm = reinterpret_cast<const int4 *>(cols + a.col0 + n0);
                int ea = 0;
                if constexpr (F64) ea = __ldg(&pscale[(int64_t)(a.cf + jj) * n_co + a.cfp + jjp].exp);
                // two columns' destinations are fetched together
#pragma unroll
                for (int c0 = 0; c0 < ECOLS; c0 += 2) {
                    int4 d0[2], d1[2];
                    int eb[2];
#pragma unroll
                    for (int u = 0; u < 2; ++u)
                        if (n0 + c0 + u < a.N) {
                            d0[u] = __ldg(cm + 2 * (c0 + u));
                            d1[u] = __ldg(cm + 2 * (c0 + u) + 1);
                            if constexpr (F64) eb[u] = __ldg(&cscale[a.coef_row0 + n0 + c0 + u].exp);
                        }
                    float vh[2] = {}, vl[2] = {};
                    if constexpr (!F64) {
                        f2_unpack(hi[c0 / 2], vh[0], vh[1]);
                        f2_unpack(lo[c0 / 2], vl[0], vl[1]);
                    }
#pragma unroll
                    for (int u = 0; u < 2; ++u) {
                        const int c = c0 + u;
                        if (n0 + c < a.N && jj - jjp >= d1[u].y) {
                            double v;
                            if constexpr (F64) v = int_words_to_double(wd[0][c], wd[1][c], ea, eb[u]);
                            else v = df_sum(vh[u], vl[u]);
                            const int64_t ld = d1[u].x;
                            double *lower = reinterpret_cast<double *>(((uint64_t)(uint32_t)d0[u].y << 32) | (uint32_t)d0[u].x);
                            double *upper = reinterpret_cast<double *>(((uint64_t)(uint32_t)d0[u].w << 32) | (uint32_t)d0[u].z);
                            lower[jj * ld + jjp] = v;
                            upper[jjp * ld + jj] = v;
                        }
                    }
                }
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TCOLS) : "memory");
    }
}

// The weak elements of an FP64 build summed in FP64 after the digits: a warp takes
// 32 rows (orbital pairs, one a lane) x 32 columns, and of those up to four elements
// of a column at a time, a lane every 32nd label in their order, so that the sums do
// not depend on which labels a symmetry-blocked panel leaves out.  digit_blk: the
// first tile of every task in the digits' launch, of whose tiles this shard takes
// every shard_n-th.  It reads a bit an element; were all elements weak, 22500 pairs x
// 210 columns over 1367 labels, it would take 15.5 ms, bound by the FP64 pipe, which
// takes 14.0 for all sums.
__global__ void __launch_bounds__(256)
fp64_elements_kernel(const SplitTask *__restrict__ tasks, const int64_t *__restrict__ blk, int n_tasks,
                     const int64_t *__restrict__ digit_blk, const uint32_t *__restrict__ weak,
                     const double *__restrict__ panel, int n_co, int Kc, int K, const int32_t *__restrict__ by_lane,
                     const ExpCol *__restrict__ all_cols, int shard_r, int shard_n) {
    constexpr unsigned full = 0xffffffffu;
    const int ti = task_of(blk, n_tasks, blockIdx.x), lane = threadIdx.x & 31;
    const SplitTask &T = tasks[ti];
    const int64_t rows = (int64_t)T.cn * T.cnp, padded = (rows + 31) / 32 * 32;
    const int64_t i = (blockIdx.x - blk[ti]) * (int64_t)256 + threadIdx.x;
    const int w = (int)(i / padded);               // the same in a warp
    const int64_t row = i % padded;
    if (w >= T.weak_words) return;
    const int jj = (int)(row / T.cnp), jjp = (int)(row % T.cnp);
    uint32_t todo = row < rows && T.cf + jj != T.cfp + jjp ? weak[T.weak0 + w * rows + row] : 0;
    const int nc = T.N - 32 * w;
    todo &= nc >= 32 ? ~0u : (1u << nc) - 1u;
    uint32_t any = __reduce_or_sync(full, todo);
    if (any == 0) return;
    const int tile_m = (jj / (BM >> T.bjp_log2)) * T.jpt_tiles + (jjp >> T.bjp_log2);
    const unsigned long long mine = (unsigned long long)(panel + ((int64_t)(T.cf + jj) * n_co + T.cfp + jjp) * Kc);
    // this lane's labels (and their panel columns): every 32nd, or those of them that
    // the block's class holds
    const int cls = T.kc0 * 64 / Kc;
    const int l0 = by_lane ? __ldg(by_lane + cls * 33 + lane) : 0;
    const int n_lab = by_lane ? __ldg(by_lane + cls * 33 + lane + 1) - l0 : (K - lane + 31) / 32;
    const int2 *__restrict__ mine_lab =
        by_lane ? reinterpret_cast<const int2 *>(by_lane + 8 * 33) + (int64_t)cls * Kc + l0 : nullptr;
    while (any) {
        const int c = 32 * w + __ffs(any) - 1;
        unsigned left = __ballot_sync(full, ((todo >> (__ffs(any) - 1)) & 1u) &&
                                                (digit_blk[ti] + (int64_t)tile_m * T.ntn + c / T.bn) % shard_n == shard_r);
        any &= any - 1;
        const ExpCol e = all_cols[T.col0 + c];
        while (left) {
            int src[4], n = 0;
            const double *p[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                src[u] = left ? __ffs(left) - 1 : src[0];
                n += left != 0;
                left &= left - 1;
                p[u] = (const double *)__shfl_sync(full, mine, src[u]);
            }
            double v[4] = {0.0, 0.0, 0.0, 0.0};
            // the loads of four labels are in flight together
            for (int i0 = 0; i0 < n_lab; i0 += 4) {
                double a[4], x[4][4];
#pragma unroll
                for (int t = 0; t < 4; ++t) {
                    const int i = i0 + t;
                    const int2 kl = i >= n_lab ? make_int2(0, 0) : (mine_lab ? __ldg(mine_lab + i) : make_int2(lane + 32 * i, lane + 32 * i));
                    a[t] = i < n_lab ? __ldg(e.arow + kl.y) : 0.0;
#pragma unroll
                    for (int u = 0; u < 4; ++u) x[t][u] = i < n_lab && u < n ? __ldg(p[u] + kl.x) : 0.0;
                }
#pragma unroll
                for (int t = 0; t < 4; ++t)
#pragma unroll
                    for (int u = 0; u < 4; ++u)
                        if (u < n && i0 + t < n_lab) v[u] = fma(x[t][u], a[t], v[u]);
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
#pragma unroll
                for (int o = 16; o; o >>= 1) v[u] += __shfl_xor_sync(full, v[u], o);
                if (u < n && lane == src[u] && jj - jjp >= e.jmin) {
                    e.lower[(int64_t)jj * e.ld + jjp] = v[u];
                    e.upper[(int64_t)jjp * e.ld + jj] = v[u];
                }
            }
        }
    }
}

// ------------------------------------------- dense split GEMM (Davidson)
// part[z][n][m] = sum over the K blocks of split z of A[m][k] X[n][k], for the
// Davidson block products H V: A (rows m of the Hamiltonian) and X (rows n =
// the block's vectors) as bf16 slices with their row exponents folded in,
// the same exact slice-pair accumulation as the expansion kernel; the K
// dimension is split over blockIdx.z (one exact chunk each) and the
// double-float partials are summed in a fixed order by dense_reduce_kernel.
struct DenseArgs {
    int M, N;                  // rows of A and of X
    int kb_total, kb_per_split;
    int a_planes, b_planes;    // K blocks per slice plane of A and of X
    float2 *part;              // [nsplit][N][M]
    int *err;
};

template <int S>
__global__ void __launch_bounds__(NTHREADS, 1)
dense_split_kernel(const __grid_constant__ CUtensorMap tm_a, const __grid_constant__ CUtensorMap tm_b, DenseArgs a) {
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    uint8_t *base = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint8_t *slots = base;
    uint64_t *full_bar = (uint64_t *)(base + S * SLOT);
    uint64_t *empty_bar = full_bar + MAXS;
    uint64_t *acc_full = empty_bar + MAXS;
    uint64_t *acc_empty = acc_full + 1;
    uint64_t *final_bar = acc_empty + 1;
    uint32_t *tmem_slot = (uint32_t *)(final_bar + 1);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int n0 = blockIdx.x * BN, m0 = blockIdx.y * BM, z = blockIdx.z;
    const int kb0 = z * a.kb_per_split;
    const int kb1 = min(a.kb_total, kb0 + a.kb_per_split);
    const int nkb = kb1 - kb0;
    const int kb_per_chunk = KCHUNK / BKB;
    const int nchunks = (nkb + kb_per_chunk - 1) / kb_per_chunk;
    int *err = a.err;
    if (threadIdx.x == 0) {
        for (int i = 0; i < MAXS; ++i) { mbar_init(&full_bar[i], 1); mbar_init(&empty_bar[i], 1); }
        mbar_init(acc_full, 1);
        mbar_init(acc_empty, EPI_THREADS);
        mbar_init(final_bar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                     "r"(TMEM_COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    if (warp == 0) {
        // TMA producer (kk: K block within this split, for slot parity and phases)
        if (lane == 0) {
            int kk = 0;
            bool ok = true;
            for (; kk < nkb && ok; ++kk) {
                const int kb = kb0 + kk;
                for (int t = 0; t < S && ok; ++t) {
                    const int sl = (kk & 1) ? slot_of<S>(1, t) : t;
                    if (kk > 0) ok = mbar_wait(&empty_bar[sl], (kk - 1) & 1, err, 1);
                    if (!ok) break;
                    uint8_t *sA = slots + sl * SLOT;
                    mbar_expect_tx(&full_bar[sl], (uint32_t)SLOT);
                    tma_load_3d(sA, &tm_a, &full_bar[sl], 0, m0, t * a.a_planes + kb);
                    tma_load_3d(sA + A_TILE, &tm_b, &full_bar[sl], 0, n0, t * a.b_planes + kb);
                }
            }
            if (kk > 0)
                for (int sl = 0; sl < S; ++sl) mbar_wait(&full_bar[sl], (kk - 1) & 1, err, 2);
        }
    } else if (warp == 1) {
        // MMA issuer
        if (lane == 0) {
            const uint32_t idesc = instr_desc_bf16(BM, BN);
            const uint64_t desc0 = smem_desc_sw128(smem_u32(slots));
            bool ok = true;
            int kk = 0;
            for (int c = 0; c < nchunks && ok; ++c) {
                if (c > 0) ok = mbar_wait(acc_empty, (c - 1) & 1, err, 3);
                if (!ok) break;
                tc_fence_after();
                const int kk_end = min(nkb, (c + 1) * kb_per_chunk);
                uint32_t fresh = 0xFu;
                for (; kk < kk_end && ok; ++kk) {
                    if (kk & 1) ok = mma_block<S, 1>(full_bar, empty_bar, 1u, tmem, desc0, idesc, fresh, err);
                    else ok = mma_block<S, 0>(full_bar, empty_bar, 0u, tmem, desc0, idesc, fresh, err);
                }
                if (ok) mma_commit(acc_full);
            }
            mma_commit(final_bar);
            mbar_wait(final_bar, 0, err, 5);
        }
    } else {
        // epilogue: rows m of A = TMEM lanes, columns = vectors n
        const int ew = warp - 2;
        const int q = warp & 3;
        const int col0 = (ew >> 2) * EPI_COLS;
        const int row = q * 32 + lane;
        f2 hi[EPI_COLS / 2], lo[EPI_COLS / 2];
#pragma unroll
        for (int c = 0; c < EPI_COLS / 2; ++c) { hi[c] = f2_pack(0.0f, 0.0f); lo[c] = f2_pack(0.0f, 0.0f); }
        bool ok = true;
        for (int c = 0; c < nchunks && ok; ++c) {
            ok = mbar_wait(acc_full, c & 1, err, 6);
            if (!ok) break;
            tc_fence_after();
            drain_chunk<S>(tmem + ((uint32_t)(q * 32) << 16) + col0, BN, hi, lo);
            tc_fence_before();
            mbar_arrive(acc_empty);
        }
        const int m = m0 + row;
        if (ok && m < a.M) {
            float2 *out = a.part + (int64_t)z * a.N * a.M + m;
#pragma unroll
            for (int c = 0; c < EPI_COLS; c += 2) {
                const int n = n0 + col0 + c;
                float h0, h1, l0, l1;
                f2_unpack(hi[c / 2], h0, h1);
                f2_unpack(lo[c / 2], l0, l1);
                if (n < a.N) out[(int64_t)n * a.M] = make_float2(h0, l0);
                if (n + 1 < a.N) out[(int64_t)(n + 1) * a.M] = make_float2(h1, l1);
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS) : "memory");
    }
}

// Y[n][m] (row stride ldy) = sum over the splits, in order, of part[z][n][m].
__global__ void dense_reduce_kernel(const float2 *__restrict__ part, int nsplit, int M, int N, double *__restrict__ Y,
                                    int64_t ldy) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= (int64_t)M * N) return;
    const int n = (int)(t / M), m = (int)(t % M);
    float h = 0.0f, l = 0.0f;
    for (int z = 0; z < nsplit; ++z) {
        const float2 x = part[((int64_t)z * N + n) * M + m];
        df_add2(h, l, x.x, x.y);
    }
    Y[(int64_t)n * ldy + m] = df_to_double(h, l);
}

// Exponent e of an FP64 bit pattern, |x| in [2^(e-1), 2^e); zeros (and FP64
// subnormals, taken as zero) give -2000, values that are not finite 1025.
__device__ __forceinline__ int fp64_exponent(unsigned long long b) {
    const int be = (int)((b >> 52) & 0x7FF);
    return be == 0 ? -2000 : be - 1022;
}

// Balanced digits of x against a row exponent: first + step (S - 1) bits in
// all, F = x 2^(bits - emax) rounded to nearest, the first digit of `first`
// bits (|d| <= 2^first), the others of `step` (|d| <= 2^(step - 1)).  put(i, d)
// takes digit i, the slice's value being d 2^(emax - first - step i).
template <class Put>
__device__ __forceinline__ void digits(double x, int emax, int S, int first, int step, Put put) {
    long long F = 0;
    if (emax > -2000) {
        const unsigned long long b = (unsigned long long)__double_as_longlong(x);
        const int be = (int)((b >> 52) & 0x7FF);
        if (be != 0) {
            const long long m = (long long)((b & 0xFFFFFFFFFFFFFull) | (1ull << 52));   // x = m 2^(be-1075)
            const int sh = (be - 1075) + first + step * (S - 1) - emax;
            long long f;
            if (sh >= 0) f = m << sh;                       // at most 62 bits
            else if (sh > -63) f = (m + (1ll << (-sh - 1))) >> (-sh);
            else f = 0;
            F = (b >> 63) ? -f : f;
        }
    }
#pragma unroll
    for (int i = 0; i < MAXS + 1; ++i) {
        if (i >= S) break;
        const int sh = step * (S - 1 - i);
        const long long d = sh > 0 ? ((F + (1ll << (sh - 1))) >> sh) : F;   // nearest digit
        F -= d << sh;
        put(i, __int_as_float(0x4B400000 + (int)d) - 12582912.0f);   // |d| < 2^22, exactly
    }
}

// Digit sizes of the expansion's slices, and of the Davidson products'.
constexpr int kXFirst = 8, kXStep = 9, kDFirst = 7, kDStep = 7;

// d 2^e for a digit d (at most 9 bits) and the exponent e of its slice; the
// result, being exact in bf16, is its upper 16 bits.
__device__ __forceinline__ uint32_t slice_bits(float d, int e) {
    if (e >= -126 && e <= 100) return __float_as_uint(d * __int_as_float((e + 127) << 23)) >> 16;
    return __bfloat16_as_ushort(__float2bfloat16_rn(ldexpf(d, e)));
}

// Magnitude of x against a row exponent as a bf16: the leading 8 bits of |x| / 2^emax,
// rounded down, in units of 2^-8; 2^-40 where they are zero and x is not, or where a
// value of the row is not finite.
__device__ __forceinline__ uint32_t magnitude_bits(double x, int emax) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(x);
    if ((b << 1) == 0) return 0;
    const int be = (int)((b >> 52) & 0x7FF), sh = 1075 - 8 - be + emax;      // 45 or more
    const unsigned long long m = (b & 0xFFFFFFFFFFFFFull) | (1ull << 52);
    const uint32_t top = be != 0 && emax > -2000 && emax <= 1024 && sh < 64 ? (uint32_t)(m >> sh) : 0;
    return top ? slice_bits((float)top, -8) : (127 - 40) << 7;
}

// Whether x is not zero, without FP64 arithmetic.
__device__ __forceinline__ int nonzero(double x) { return ((unsigned long long)__double_as_longlong(x) << 1) != 0; }

// The scale of a row with exponent emax and nz entries that are not zero.  The line is
// half-way between two sums of magnitudes, which are multiples of 2^-16 but for the
// 2^-40 ones, so that the order in which they are added does not matter.
__device__ __forceinline__ RowScale row_scale(int emax, int nz) {
    const float at = fmaxf(sqrtf((float)nz) / 512.0f, 1.0f / 128.0f);
    return {emax > 1024 ? kExpNaN : (emax > -2000 ? emax : 0), (floorf(at * 65536.0f) + 0.5f) / 65536.0f};
}

// One row into its S bf16 slices by a whole block: every thread reads its
// share of the row, the row exponent is reduced through shared memory, then
// each thread writes the digits of its elements, two neighbours to a store.
// at(k) gives element k (0 beyond the row's data).  With SCALES the row's goes to
// `scales`, the slices are those of x / 2^e, and slice S holds the magnitudes.
// (Decided at compile time: left to the pointer, the count of the entries and the
// magnitudes, which mixed builds have not, made theirs slower too: a batch of 12
// over 8 symmetries 3.71 ms, 3.62 without.)
template <bool SCALES, class At>
__device__ __forceinline__ void slice_row_block(At at, int64_t dest, int64_t R, int Kpad, int S, int first, int step,
                                                __nv_bfloat16 *__restrict__ out, RowScale *__restrict__ scales = nullptr) {
    __shared__ int red[32], count[SCALES ? 32 : 1];
    int emax = -2000, nz = 0;
    for (int k = 2 * threadIdx.x; k < Kpad; k += 2 * blockDim.x) {
        const double x0 = at(k), x1 = at(k + 1);
        emax = max(emax, max(fp64_exponent((unsigned long long)__double_as_longlong(x0)),
                             fp64_exponent((unsigned long long)__double_as_longlong(x1))));
        if (SCALES) nz += nonzero(x0) + nonzero(x1);
    }
#pragma unroll
    for (int off = 16; off; off >>= 1) emax = max(emax, __shfl_xor_sync(0xffffffffu, emax, off));
    if (SCALES) nz = __reduce_add_sync(0xffffffffu, nz);
    const int warp = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
    if ((threadIdx.x & 31) == 0) {
        red[warp] = emax;
        if (SCALES) count[warp] = nz;
    }
    __syncthreads();
    emax = -2000;
    nz = 0;
    for (int w = 0; w < nw; ++w) {
        emax = max(emax, red[w]);
        if (SCALES) nz += count[w];
    }
    if (SCALES && threadIdx.x == 0) scales[dest] = row_scale(emax, nz);
    const int64_t plane = (int64_t)(Kpad / BKB) * R * BKB;
    const int e0 = SCALES ? 0 : emax;
    for (int k = 2 * threadIdx.x; k < Kpad; k += 2 * blockDim.x) {
        uint32_t *o = reinterpret_cast<uint32_t *>(out + ((int64_t)(k / BKB) * R + dest) * BKB + k % BKB);
        uint32_t lo[MAXS + 1];
        digits(at(k), emax, S, first, step, [&](int i, float d) { lo[i] = slice_bits(d, e0 - first - step * i); });
        digits(at(k + 1), emax, S, first, step, [&](int i, float d) {
            o[i * (plane / 2)] = lo[i] | slice_bits(d, e0 - first - step * i) << 16;
        });
        if (SCALES) o[S * (plane / 2)] = magnitude_bits(at(k), emax) | magnitude_bits(at(k + 1), emax) << 16;
    }
}

// Rows of [X1 | X2] (K1 then K2 entries, row strides ld1, ld2; X2 may be
// absent) into bf16 slices [S][Kpad/64][R][64], one block per row.
__global__ void __launch_bounds__(1024)
slice_rows2_kernel(const double *__restrict__ X1, int64_t ld1, int K1, const double *__restrict__ X2, int64_t ld2,
                   int K2, int Kpad, int S, int64_t R, __nv_bfloat16 *__restrict__ out) {
    const int64_t row = blockIdx.x;
    const double *x1 = X1 + row * ld1;
    const double *x2 = X2 ? X2 + row * ld2 : nullptr;
    slice_row_block<false>([&](int k) -> double { return k < K1 ? __ldg(x1 + k) : ((x2 && k < K1 + K2) ? __ldg(x2 + k - K1) : 0.0); },
                    row, R, Kpad, S, kDFirst, kDStep, out);
}

// ------------------------------------------------------------- slicing
// One warp per row (as slice_row_block).  Output layout [S][K/64][R][64] (R rows
// in all), so a 64-wide K block of consecutive rows is contiguous.  Column
// skip_col is zero.
__device__ __forceinline__ void slice_row(const double *__restrict__ x, int64_t dest, int64_t R, int Kpad, int S,
                                          int skip_col, __nv_bfloat16 *__restrict__ out, RowScale *__restrict__ scales,
                                          int lane) {
    const int KB = Kpad / BKB;
    // exponent of the row maximum from the bit patterns (no FP64 arithmetic)
    int emax = -2000;
    for (int k = lane; k < Kpad; k += 32)
        if (k != skip_col) emax = max(emax, fp64_exponent((unsigned long long)__double_as_longlong(x[k])));
#pragma unroll
    for (int off = 16; off; off >>= 1) emax = max(emax, __shfl_xor_sync(0xffffffffu, emax, off));
    if (scales) {
        int nz = 0;
        for (int k = lane; k < Kpad; k += 32) nz += k != skip_col && nonzero(x[k]);
        nz = __reduce_add_sync(0xffffffffu, nz);
        if (lane == 0) scales[dest] = row_scale(emax, nz);
    }
    const int e0 = scales ? 0 : emax;
    for (int k = lane; k < Kpad; k += 32) {
        const int kb = k / BKB, kk = k % BKB;
        digits(k != skip_col ? x[k] : 0.0, emax, S, kXFirst, kXStep, [&](int i, float d) {
            out[(((int64_t)i * KB + kb) * R + dest) * BKB + kk] =
                __ushort_as_bfloat16((unsigned short)slice_bits(d, e0 - kXFirst - kXStep * i));
        });
        if (scales)
            out[(((int64_t)S * KB + kb) * R + dest) * BKB + kk] =
                __ushort_as_bfloat16((unsigned short)(k != skip_col ? magnitude_bits(x[k], emax) : 0));
    }
}

// Panel rows (j n_co + j') into slices; column skip_col (the delta label) is
// zeroed on the rows with j == j' (elsewhere that label is zero, or, with
// orbital symmetry, the column holds another label).
__global__ void slice_rows_kernel(const double *__restrict__ X, int64_t rows, int Kpad, int S, int skip_col,
                                  int n_co, __nv_bfloat16 *__restrict__ out, RowScale *__restrict__ scales) {
    const int64_t row = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (row >= rows) return;
    const bool diag = row / n_co == row % n_co;
    slice_row(X + row * Kpad, row, rows, Kpad, S, diag ? skip_col : -1, out, scales, threadIdx.x & 31);
}

// Coefficient rows (Kin entries each) into slices of Kout columns: column k
// holds label perm[k] (the labels class by class, with orbital symmetry; -1
// padding), or label k without a permutation; column skip_col (the delta
// label) is zero.
template <bool SCALES>
__global__ void __launch_bounds__(256)
slice_rows_grouped(const SliceTask *__restrict__ tasks, const int64_t *__restrict__ blk, int n_tasks, int64_t R,
                   int Kin, int Kout, const int32_t *__restrict__ perm, int S, int skip_col,
                   __nv_bfloat16 *__restrict__ out, RowScale *__restrict__ scales) {
    const int ti = task_of(blk, n_tasks, blockIdx.x);
    const SliceTask &T = tasks[ti];
    const int64_t row = blockIdx.x - blk[ti];
    const double *x = T.X + row * Kin;
    slice_row_block<SCALES>([&](int k) -> double {
        if (k == skip_col) return 0.0;
        const int lab = perm ? __ldg(perm + k) : k;
        return (lab >= 0 && lab < Kin) ? __ldg(x + lab) : 0.0;
    }, T.row0 + row, R, Kout, S, kXFirst, kXStep, out, scales);
}

// Rows with j == j' (both ranges): H[(n,j),(n',j)] over all K, incl. delta,
// in double-float (they carry h_jj and the delta_jj' E term and so have a
// wide dynamic range that the bf16 slices of one row do not cover).  Per task
// one block per (j, 8 state pairs); the lanes of a warp split K.
// A block computes a tile of kDRj rows j x kDRt coefficient rows t; the
// panel and coefficient rows pass through shared memory in K-chunks (the next
// chunk is read into registers while the current one is used) and every
// thread keeps four double-float partial sums (k mod 4), combined in a fixed
// order at the end.
constexpr int kDRj = 16, kDRt = 16, kDRk = 128;
constexpr int kDRthreads = kDRj * kDRt;
constexpr int kDRper = kDRj * kDRk / kDRthreads;     // elements of each tile a thread moves per chunk

__global__ void __launch_bounds__(kDRthreads)
diag_rows_kernel(const DRTask *__restrict__ tasks, const int64_t *__restrict__ blk, int n_tasks) {
    static_assert(kDRj == kDRt, "both tiles are moved by the same index pattern");
    __shared__ float2 sp[kDRj][kDRk + 1], sa[kDRt][kDRk + 1];
    const int ti = task_of(blk, n_tasks, blockIdx.x);
    const DRTask &T = tasks[ti];
    const int lb = (int)(blockIdx.x - blk[ti]);
    const int j0 = T.j_lo + (lb / T.ny) * kDRj, t0 = (lb % T.ny) * kDRt;
    const int tl = threadIdx.x % kDRt, jl = threadIdx.x / kDRt;
    const int j = j0 + jl, t = t0 + tl;
    const int Kpad = T.Kpad, Ka = T.Ka, j_hi = T.j_hi, n_nn = T.n_nn;
    const float2 *__restrict__ Pd = T.Pd;
    const float2 *__restrict__ A = T.A;
    const int32_t *__restrict__ perm = T.perm;
    float2 rp[kDRper], ra[kDRper];
    auto fetch = [&](int k0) {
#pragma unroll
        for (int u = 0; u < kDRper; ++u) {
            const int i = threadIdx.x + u * kDRthreads;
            const int r = i / kDRk, k = k0 + i % kDRk;
            const bool kin = k < Kpad;
            rp[u] = (kin && j0 + r < j_hi) ? __ldg(Pd + (int64_t)(j0 + r) * Kpad + k) : make_float2(0.0f, 0.0f);
            const int lab = (kin && perm) ? __ldg(perm + k) : k;   // the label of panel column k
            ra[u] = (kin && lab >= 0 && t0 + r < n_nn) ? __ldg(A + (int64_t)(t0 + r) * Ka + lab)
                                                        : make_float2(0.0f, 0.0f);
        }
    };
    float h[4] = {0.0f, 0.0f, 0.0f, 0.0f}, l[4] = {0.0f, 0.0f, 0.0f, 0.0f};
    fetch(0);
    for (int k0 = 0; k0 < Kpad; k0 += kDRk) {
        __syncthreads();
#pragma unroll
        for (int u = 0; u < kDRper; ++u) {
            const int i = threadIdx.x + u * kDRthreads;
            sp[i / kDRk][i % kDRk] = rp[u];
            sa[i / kDRk][i % kDRk] = ra[u];
        }
        __syncthreads();
        if (k0 + kDRk < Kpad) fetch(k0 + kDRk);
#pragma unroll 2
        for (int k = 0; k < kDRk; k += 4) {
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const float2 x = sp[jl][k + u], y = sa[tl][k + u];
                df_fma(h[u], l[u], x.x, x.y, y.x, y.y);
            }
        }
    }
    if (j >= j_hi || t >= n_nn) return;
    df_add2(h[0], l[0], h[1], l[1]);
    df_add2(h[2], l[2], h[3], l[3]);
    df_add2(h[0], l[0], h[2], l[2]);
    const int na = T.nn[2 * t], nb = T.nn[2 * t + 1];
    const int64_t r = T.row_off + (int64_t)na * T.cn + (j - T.cf);
    const int64_t c = T.col_off + (int64_t)nb * T.cnp + (j - T.cfp);
    if (T.same && r < c) return;
    const double v = df_to_double(h[0], l[0]);
    T.H[r * T.ld + c] = v;
    if (r != c) T.H[c * T.ld + r] = v;
}

// The same in FP64, for the FP64 build: a thread adds one element's labels in
// their order, so the sums do not depend on which labels a symmetry-blocked
// panel leaves out (their terms are zero).  150 rows x 210 pairs x 1367 labels
// hold the FP64 pipe for 68 us.
constexpr int kD64k = 32;
__global__ void __launch_bounds__(kDRthreads)
diag_rows_f64_kernel(const DRTask *__restrict__ tasks, const int64_t *__restrict__ blk, int n_tasks) {
    __shared__ double sp[kDRj][kD64k + 1], sa[kDRt][kD64k + 1];
    const int ti = task_of(blk, n_tasks, blockIdx.x);
    const DRTask &T = tasks[ti];
    const int lb = (int)(blockIdx.x - blk[ti]);
    const int j0 = T.j_lo + (lb / T.ny) * kDRj, t0 = (lb % T.ny) * kDRt;
    const int tl = threadIdx.x % kDRt, jl = threadIdx.x / kDRt;
    const int j = j0 + jl, t = t0 + tl;
    constexpr int per = kDRj * kD64k / kDRthreads;
    double rp[per], ra[per];
    auto fetch = [&](int k0) {
#pragma unroll
        for (int u = 0; u < per; ++u) {
            const int i = threadIdx.x + u * kDRthreads;
            const int r = i / kD64k, k = k0 + i % kD64k;
            const bool kin = k < T.Kpad;
            const int lab = (kin && T.perm) ? __ldg(T.perm + k) : k;   // the label of panel column k
            rp[u] = (kin && j0 + r < T.j_hi) ? __ldg(T.P64 + ((int64_t)(j0 + r) * T.n_co + j0 + r) * T.Kpad + k) : 0.0;
            ra[u] = (kin && lab >= 0 && t0 + r < T.n_nn) ? __ldg(T.A64 + (int64_t)(t0 + r) * T.Ka + lab) : 0.0;
        }
    };
    double v = 0.0;
    fetch(0);
    for (int k0 = 0; k0 < T.Kpad; k0 += kD64k) {
        __syncthreads();
#pragma unroll
        for (int u = 0; u < per; ++u) {
            const int i = threadIdx.x + u * kDRthreads;
            sp[i / kD64k][i % kD64k] = rp[u];
            sa[i / kD64k][i % kD64k] = ra[u];
        }
        __syncthreads();
        if (k0 + kD64k < T.Kpad) fetch(k0 + kD64k);
#pragma unroll 8
        for (int k = 0; k < kD64k; ++k) v = fma(sp[jl][k], sa[tl][k], v);
    }
    if (j >= T.j_hi || t >= T.n_nn) return;
    const int na = T.nn[2 * t], nb = T.nn[2 * t + 1];
    const int64_t r = T.row_off + (int64_t)na * T.cn + (j - T.cf);
    const int64_t c = T.col_off + (int64_t)nb * T.cnp + (j - T.cfp);
    if (T.same && r < c) return;
    T.H[r * T.ld + c] = v;
    if (r != c) T.H[c * T.ld + r] = v;
}

// Diagonal panel rows P[(j, j)][k] as float pairs.
__global__ void panel_diag_df_kernel(const double *__restrict__ P, int n_co, int Kpad, float2 *__restrict__ out) {
    const int j = blockIdx.x;
    for (int k = threadIdx.x; k < Kpad; k += blockDim.x) {
        const double v = P[((int64_t)j * n_co + j) * Kpad + k];
        const float h = (float)v;
        out[(int64_t)j * Kpad + k] = make_float2(h, (float)(v - (double)h));
    }
}

// ------------------------------------------------------ tensor maps (host)
typedef CUresult (*EncodeTiled)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiled encode_fn() {
    static EncodeTiled fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = (EncodeTiled)p;
    });
    return fn;
}

}  // namespace

// dynamic shared memory of the expansion kernel: the operand slots, the
// barriers and the 1 KB alignment
static int split_smem_bytes(int bn, int ks, int slots = 0) {
    return (slots ? slots : xslots(bn, ks)) * xslot(bn, ks) + 1024 + (2 * XBARS + 2 * XACC + 2) * 8;
}

static int sm_count() {
    static int n = 0;
    if (n == 0) {
        int dev = 0, v = 0;
        if (cudaGetDevice(&dev) == cudaSuccess &&
            cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess && v > 0)
            n = v;
        else
            n = 1;
    }
    return n;
}

template <int S, int MODE>
static cudaError_t set_smem_attr_s() {
    const auto attr = cudaFuncAttributeMaxDynamicSharedMemorySize;
    cudaError_t e = cudaFuncSetAttribute(split_expand_kernel<S, 32, 32, MODE>, attr, split_smem_bytes(32, 32));
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(split_expand_kernel<S, 64, 32, MODE>, attr, split_smem_bytes(64, 32));
    if constexpr (MODE == kMixedSums) {
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(split_expand_kernel<S, 128, 32, MODE>, attr, split_smem_bytes(128, 32));
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(split_expand_kernel<S, 128, 64, MODE>, attr, split_smem_bytes(128, 64));
    } else if (e == cudaSuccess) {
        e = cudaFuncSetAttribute(split_expand_kernel<1, kWeakCols, 64, kWeakBits>, attr,
                                 split_smem_bytes(kWeakCols, 64, kWeakSlots));
    }
    return e;
}

static cudaError_t set_smem_attr(int S) {
    switch (S) {
        case 2: return set_smem_attr_s<2, kMixedSums>();
        case 3: return set_smem_attr_s<3, kMixedSums>();
        case 4: return set_smem_attr_s<4, kMixedSums>();
        case 5: return set_smem_attr_s<5, kMixedSums>();
        case 6: return set_smem_attr_s<6, kMixedSums>();
        default: return set_smem_attr_s<kF64Slices, kF64Sums>();
    }
}

static int mixed_fail(hb_ctx *ctx, int code, const std::string &m) {
    ctx->err = m;
    return code;
}

// The slices of an FP64 build are 16 bytes for every 8 of the panel, and it can do
// without them: outside a caller's workspace (sized with them or not) they take
// no more than a quarter of the memory that is free, so that the caller, other
// contexts and the solve find most of what they found before.  (An eighth would
// leave out a batch over 2513 continuum orbitals, 32 GB of slices beside 235 GB of
// free memory, which takes 20 ms with them and 280 without.)
bool f64_slices_fit(const hb_ctx *ctx, size_t bytes) {
    if (ctx->pool.base) return true;
    size_t free = 0, total = 0;
    if (cudaMemGetInfo(&free, &total) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return bytes <= free / 4;
}

// Panel slices and their tensor maps, once per context and precision (the
// integrals do not change between builds); a context that borrows its
// integrals borrows these.
int mixed_prepare(hb_ctx *ctx, int precision, cudaStream_t s) {
    if (!ctx->mixed) ctx->mixed = new MixedState();
    MixedState &M = *ctx->mixed;
    PanelSlices &PS = M.panel[precision == HB_MIXED];
    if (PS.ready) return HB_OK;
    if (ctx->base) {
        int rc = mixed_prepare(ctx->base, precision, s);
        if (rc != HB_OK) return mixed_fail(ctx, rc, ctx->base->err);
        PS = ctx->base->mixed->panel[precision == HB_MIXED];
        PS.borrowed = true;
        if (precision == HB_MIXED) M.pdiag = ctx->base->mixed->pdiag;
        return HB_OK;
    }
    PS.slices = precision == HB_MIXED ? ctx->expand_slices : kF64Slices;
    if (precision == HB_MIXED && (PS.slices < 2 || PS.slices > MAXS))
        return mixed_fail(ctx, HB_ERR_INVALID_ARG, "split_slices must be 2..6");
    if (!encode_fn()) return mixed_fail(ctx, HB_ERR_CUDA, "cuTensorMapEncodeTiled is not available");
    const int64_t rows = (int64_t)ctx->n_co * ctx->n_co;
    // the panel's columns: every label, or with orbital symmetry the Kc labels
    // of each row's class
    const int Kc = ctx->Kc;
    const int planes = precision == HB_FP64 ? kF64Planes : PS.slices;
    const size_t bytes = sizeof(__nv_bfloat16) * (size_t)planes * rows * Kc;
    if (precision == HB_FP64 && !f64_slices_fit(ctx, bytes))
        return mixed_fail(ctx, HB_ERR_OOM, "panel slices: more than an FP64 build may take");
    const size_t extra = precision == HB_MIXED ? sizeof(float2) * (size_t)ctx->n_co * Kc : sizeof(RowScale) * (size_t)rows;
    // everything that can fail comes before the kernels; a failure leaves nothing behind
    auto undo = [&](int code, const std::string &m) {
        dfree(ctx, PS.buf);
        dfree(ctx, PS.scales);
        PS.buf = nullptr;
        PS.scales = nullptr;
        if (precision == HB_MIXED) {
            dfree(ctx, M.pdiag);
            M.pdiag = nullptr;
        }
        return mixed_fail(ctx, code, m);
    };
    cudaError_t e = dmalloc(ctx, (void **)&PS.buf, bytes);
    if (e == cudaSuccess) e = precision == HB_MIXED ? dmalloc(ctx, (void **)&M.pdiag, extra) : dmalloc(ctx, (void **)&PS.scales, extra);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return undo(HB_ERR_OOM, std::string("panel slices: ") + cudaGetErrorString(e));
    }
    // 4D map over the panel slices [S*KB][j][j'][64]: coordinates (kk, j', j, plane)
    const int KB = Kc / BKB;
    cuuint64_t dims[4] = {(cuuint64_t)BKB, (cuuint64_t)ctx->n_co, (cuuint64_t)ctx->n_co,
                          (cuuint64_t)planes * KB};
    cuuint64_t strides[3] = {(cuuint64_t)BKB * 2, (cuuint64_t)ctx->n_co * BKB * 2, (cuuint64_t)rows * BKB * 2};
    cuuint32_t estr[4] = {1, 1, 1, 1};
    CUresult r = CUDA_SUCCESS;
    for (int w = 0; w < 2 && r == CUDA_SUCCESS; ++w)
        for (int i = 0; i < 3 && r == CUDA_SUCCESS; ++i) {
            const int lg = 3 + i;
            // a 32-K stage copies half a 64-wide K block (x = 0 or 32: 64-byte
            // aligned, 64-byte swizzle), a 64-K stage all of it (128-byte swizzle)
            cuuint32_t box[4] = {w ? 64u : 32u, (cuuint32_t)(1 << lg), (cuuint32_t)(BM >> lg), 1};
            r = encode_fn()(&PS.tm[w][i], CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, PS.buf, dims, strides,
                            box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                            w ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B,
                            CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
        }
    if (r != CUDA_SUCCESS) return undo(HB_ERR_CUDA, "panel tensor map: error " + std::to_string((int)r));
    e = set_smem_attr(PS.slices);
    if (e != cudaSuccess) return undo(HB_ERR_CUDA, std::string("smem attribute: ") + cudaGetErrorString(e));
    ctx->dev_bytes += bytes + extra;
    if (precision == HB_MIXED) panel_diag_df_kernel<<<ctx->n_co, 256, 0, s>>>(ctx->panel, ctx->n_co, Kc, M.pdiag);
    slice_rows_kernel<<<(unsigned)((rows + 7) / 8), 256, 0, s>>>(ctx->panel, rows, Kc, PS.slices, ctx->delta_pos,
                                                                 ctx->n_co, PS.buf, PS.scales);
    PS.ready = true;
    return HB_OK;
}

const void *mixed_panel_key(const hb_ctx *ctx, int precision) {
    return ctx->mixed ? ctx->mixed->panel[precision == HB_MIXED].buf : nullptr;
}
const float2 *mixed_panel_diag(const hb_ctx *ctx) { return ctx->mixed ? ctx->mixed->pdiag : nullptr; }
int mixed_slices(const hb_ctx *ctx, int precision) {
    return precision == HB_MIXED ? (ctx->mixed ? ctx->mixed->panel[1].slices : ctx->expand_slices) : kF64Slices;
}

// Coefficient slices of `rows` rows in all: [S][Kpad/64][rows][64] bf16 and
// four 3D maps: for 32-K stages one per tile width bn = 32, 64, 128 (box: bn
// rows x half a K block of one slice plane, 64-byte swizzle), and for 64-K
// stages one of 128 rows x a whole K block (128-byte swizzle).
// scales (FP64 build, or null): those of the rows.
int split_coef_alloc(hb_ctx *mem, int S, int64_t rows, int Kpad, void **buf, RowScale **scales, CUtensorMap *tm,
                     std::string *err) {
    *buf = nullptr;
    if (scales) *scales = nullptr;
    if (!encode_fn()) { *err = "cuTensorMapEncodeTiled is not available"; return HB_ERR_CUDA; }
    if (rows < 1) rows = 1;
    cudaError_t e = dmalloc(mem, buf, sizeof(__nv_bfloat16) * (size_t)S * rows * Kpad);
    if (e == cudaSuccess && scales) e = dmalloc_n(mem, scales, (size_t)rows);
    if (e != cudaSuccess) {
        cudaGetLastError();
        dfree(mem, *buf);
        *buf = nullptr;
        *err = std::string("coefficient slices: ") + cudaGetErrorString(e);
        return HB_ERR_OOM;
    }
    const int KB = Kpad / BKB;
    cuuint64_t dims[3] = {(cuuint64_t)BKB, (cuuint64_t)rows, (cuuint64_t)S * KB};
    cuuint64_t strides[2] = {(cuuint64_t)BKB * 2, (cuuint64_t)rows * BKB * 2};
    cuuint32_t estr[3] = {1, 1, 1};
    CUresult r = CUDA_SUCCESS;
    for (int i = 0; i < 4 && r == CUDA_SUCCESS; ++i) {
        cuuint32_t box[3] = {i < 3 ? 32u : 64u, (cuuint32_t)(i < 3 ? 32 << i : 128), 1};
        r = encode_fn()(&tm[i], CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, *buf, dims, strides, box, estr,
                        CU_TENSOR_MAP_INTERLEAVE_NONE, i < 3 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_128B,
                        CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    }
    if (r != CUDA_SUCCESS) {
        dfree(mem, *buf);
        *buf = nullptr;
        if (scales) { dfree(mem, *scales); *scales = nullptr; }
        *err = "coefficient tensor map: error " + std::to_string((int)r);
        return HB_ERR_CUDA;
    }
    return HB_OK;
}

int64_t blocks_split(int cn, int cnp, int N, int lg, int bn) {
    if (cn <= 0 || cnp <= 0 || N <= 0) return 0;
    const int bj = BM >> lg, bjp = 1 << lg;
    return (int64_t)((N + bn - 1) / bn) * ((cn + bj - 1) / bj) * ((cnp + bjp - 1) / bjp);
}
int split_ntn(int N, int bn) { return (N + bn - 1) / bn; }

// Tile width for a merged block of N columns over kblocks 64-wide K blocks:
// the narrowest of 32 and 64 that holds them, else 128 (whose MMAs read the
// least shared memory per flop).  Over long K every tile is 128 wide, so that
// every tile of the plan takes the same K stage (64) and a block's bits do not
// depend on the columns it is merged with.  `force` (32, 64, 128) overrides.
int split_cols_choice(int N, int kblocks, int force) {
    if (force == 32 || force == 64 || force == 128) return force;
    if (kblocks >= kK64Blocks) return 128;
    return N <= 32 ? 32 : (N <= 64 ? 64 : 128);
}
// The FP64 kernel's seven accumulators fit tensor memory up to 64 columns; its
// sums are exact, so no shape changes a bit.
int split_f64_cols_choice(int N, int force) { return force == 32 || (force == 0 && N <= 32) ? 32 : 64; }
int split_jpt(int cnp, int lg) { return (cnp + (1 << lg) - 1) >> lg; }

// Tile arrangement with the least padding of the cn x cnp rectangle; of equal
// ones 16 x 8, whose warps (4 j x 8 j') write whole 32-byte sectors of both the
// block and its mirror.
int split_tile_heuristic(int cn, int cnp) {
    int best = 3;
    int64_t best_area = -1;
    for (int lg : {3, 4, 5}) {
        const int bj = BM >> lg, bjp = 1 << lg;
        const int64_t area = (int64_t)((cn + bj - 1) / bj) * bj * ((cnp + bjp - 1) / bjp) * bjp;
        if (best_area < 0 || area < best_area) { best = lg; best_area = area; }
    }
    return best;
}

int g_slice(const Grouped<SliceTask> &g, int64_t R, int Kin, int Kout, const int32_t *perm, int S, int skip_col,
            void *out, RowScale *scales, cudaStream_t s) {
    if (g.blocks <= 0) return 0;
    auto *kernel = scales ? slice_rows_grouped<true> : slice_rows_grouped<false>;
    kernel<<<(unsigned)g.blocks, 256, 0, s>>>(g.tasks, g.blk, g.n, R, Kin, Kout, perm, S, skip_col, (__nv_bfloat16 *)out,
                                              scales);
    return 1;
}

int split_kstage_choice(int bn, int kblocks, int force) {
    if (bn != 128) return 32;
    if (force == 32 || force == 64) return force;
    return kblocks >= kK64Blocks ? 64 : 32;
}

int g_weak_bits(const hb_ctx *panel_ctx, int lg, const CUtensorMap *tm_coef, const RowScale *coef_scales,
                const Grouped<SplitTask> &g, uint32_t *weak, int kblocks, int coef_planes, const ExpCol *cols, int *err, cudaStream_t s) {
    if (g.blocks <= 0) return 0;
    const PanelSlices &PS = panel_ctx->mixed->panel[0];
    const unsigned grid = (unsigned)std::min((int)g.blocks, sm_count());
    split_expand_kernel<1, kWeakCols, 64, kWeakBits><<<grid, NTHREADS, split_smem_bytes(kWeakCols, 64, kWeakSlots), s>>>(
        PS.tm[1][lg - 3], tm_coef[3], g.tasks, g.blk, g.n, (int)g.blocks, kblocks, coef_planes, cols, PS.scales, coef_scales,
        weak, kF64Slices, panel_ctx->n_co, err, 0, 1);
    return 1;
}

int64_t blocks_weak_sums(int cn, int cnp, int N) {
    return (((int64_t)cn * cnp + 31) / 32 * 32 * ((N + 31) / 32) + 255) / 256;
}
int g_weak_sums(const hb_ctx *panel_ctx, const Grouped<SplitTask> &g, const Grouped<SplitTask> &digits,
                const uint32_t *weak, int kblocks, const ExpCol *cols, cudaStream_t s, int shard_r, int shard_n) {
    if (g.blocks <= 0) return 0;
    fp64_elements_kernel<<<(unsigned)g.blocks, 256, 0, s>>>(
        g.tasks, g.blk, g.n, digits.blk, weak, panel_ctx->panel, panel_ctx->n_co, kblocks * 64, panel_ctx->K,
        panel_ctx->cls_by_lane, cols, shard_r, shard_n);
    return 1;
}

int g_split(const hb_ctx *panel_ctx, int precision, int lg, int bn, const CUtensorMap *tm_coef, const RowScale *coef_scales,
            const Grouped<SplitTask> &g, int kblocks, int coef_planes, const ExpCol *cols, int *err, cudaStream_t s,
            int shard_r, int shard_n) {
    if (g.blocks <= 0) return 0;
    const bool f64 = precision != HB_MIXED;
    if (bn != 32 && bn != 64 && (f64 || bn != 128)) return 0;
    const PanelSlices &PS = panel_ctx->mixed->panel[!f64];
    const int ks = f64 ? 32 : split_kstage_choice(bn, kblocks, panel_ctx->force_kstage);
    const CUtensorMap &tm_panel = PS.tm[ks == 64 ? 1 : 0][lg - 3];
    const CUtensorMap &tm_c = tm_coef[ks == 64 ? 3 : (bn == 32 ? 0 : (bn == 64 ? 1 : 2))];
    const size_t smem = split_smem_bytes(bn, ks);
    // persistent: one CTA per SM at most (each fills its SM's shared memory)
    const int n_tiles = (int)g.blocks;
    const int n_local = n_tiles > shard_r ? (n_tiles - shard_r + shard_n - 1) / shard_n : 0;
    if (n_local <= 0) return 0;
    const unsigned grid = (unsigned)std::min(n_local, sm_count());
#define HB_SPLIT(SS, BB, KK, MM)                                                                                   \
    split_expand_kernel<SS, BB, KK, MM><<<grid, NTHREADS, smem, s>>>(tm_panel, tm_c, g.tasks, g.blk, g.n, n_tiles, \
                                                                     kblocks, coef_planes, cols, PS.scales, coef_scales, \
                                                                     nullptr, 0, panel_ctx->n_co, err, shard_r, \
                                                                     shard_n)
#define HB_SPLIT_S(SS)                                       \
    do {                                                     \
        if (bn == 32) HB_SPLIT(SS, 32, 32, kMixedSums);      \
        else if (bn == 64) HB_SPLIT(SS, 64, 32, kMixedSums); \
        else if (ks == 32) HB_SPLIT(SS, 128, 32, kMixedSums);\
        else HB_SPLIT(SS, 128, 64, kMixedSums);              \
    } while (0)
    if (f64) {
        if (bn == 32) HB_SPLIT(kF64Slices, 32, 32, kF64Sums);
        else HB_SPLIT(kF64Slices, 64, 32, kF64Sums);
        return 1;
    }
    switch (PS.slices) {
        case 2: HB_SPLIT_S(2); break;
        case 3: HB_SPLIT_S(3); break;
        case 4: HB_SPLIT_S(4); break;
        case 5: HB_SPLIT_S(5); break;
        default: HB_SPLIT_S(6); break;
    }
#undef HB_SPLIT_S
#undef HB_SPLIT
    return 1;
}

int64_t blocks_diag_rows(int j_lo, int j_hi, int n_nn) {
    if (j_hi <= j_lo || n_nn <= 0) return 0;
    return (int64_t)((j_hi - j_lo + kDRj - 1) / kDRj) * ((n_nn + kDRt - 1) / kDRt);
}
int diag_rows_ny(int n_nn) { return (n_nn + kDRt - 1) / kDRt; }

int g_diag_rows(const Grouped<DRTask> &g, int dfloat, cudaStream_t s) {
    if (g.blocks <= 0) return 0;
    if (!dfloat) diag_rows_f64_kernel<<<(unsigned)g.blocks, kDRthreads, 0, s>>>(g.tasks, g.blk, g.n);
    else diag_rows_kernel<<<(unsigned)g.blocks, kDRthreads, 0, s>>>(g.tasks, g.blk, g.n);
    return 1;
}

// ------------------------------------------------ dense split GEMM (host)
int dense_operand_alloc(hb_ctx *mem, int S, int64_t R, int Kpad, DenseOperand *op, std::string *err) {
    op->buf = nullptr;
    op->R = R < 1 ? 1 : R;
    op->Kpad = Kpad;
    op->planes = Kpad / BKB;
    if (!encode_fn()) { *err = "cuTensorMapEncodeTiled is not available"; return HB_ERR_CUDA; }
    const size_t bytes = sizeof(__nv_bfloat16) * (size_t)S * op->planes * op->R * BKB;
    cudaError_t e = dmalloc(mem, (void **)&op->buf, bytes);
    if (e != cudaSuccess) { *err = std::string("Davidson operand slices: ") + cudaGetErrorString(e); return HB_ERR_OOM; }
    cuuint64_t dims[3] = {(cuuint64_t)BKB, (cuuint64_t)op->R, (cuuint64_t)S * op->planes};
    cuuint64_t strides[2] = {(cuuint64_t)BKB * 2, (cuuint64_t)op->R * BKB * 2};
    cuuint32_t box[3] = {BKB, BM, 1};
    cuuint32_t estr[3] = {1, 1, 1};
    CUresult r = encode_fn()(&op->tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, op->buf, dims, strides, box, estr,
                             CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                             CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) {
        dfree(mem, op->buf);
        op->buf = nullptr;
        *err = "Davidson operand tensor map: error " + std::to_string((int)r);
        return HB_ERR_CUDA;
    }
    return HB_OK;
}

void dense_operand_free(hb_ctx *mem, DenseOperand *op) {
    if (op->buf) dfree(mem, op->buf);
    op->buf = nullptr;
}

void dense_operand_fill(const DenseOperand &op, int S, const double *X1, int64_t ld1, int K1, const double *X2,
                        int64_t ld2, int K2, int64_t rows, cudaStream_t s) {
    if (rows <= 0) return;
    slice_rows2_kernel<<<(unsigned)rows, 1024, 0, s>>>(X1, ld1, K1, X2, ld2, K2, op.Kpad, S, op.R,
                                                       (__nv_bfloat16 *)op.buf);
}

int dense_splits(int64_t M, int64_t N, int kb_total, int *kb_per_split) {
    const int64_t tiles = ((M + BM - 1) / BM) * ((N + BN - 1) / BN);
    const int kpc = KCHUNK / BKB;
    const int max_split = (kb_total + kpc - 1) / kpc;
    int ns = (int)std::max<int64_t>(1, std::min<int64_t>(max_split, (3 * 152 + tiles - 1) / tiles));
    int per = (kb_total + ns - 1) / ns;
    per = (per + kpc - 1) / kpc * kpc;
    *kb_per_split = per;
    return (kb_total + per - 1) / per;
}

int dense_split_gemm(int S, const DenseOperand &A, int64_t M, const DenseOperand &B, int64_t N, int kb_total,
                     float2 *part, double *Y, int64_t ldy, int *err, cudaStream_t s) {
    if (M <= 0 || N <= 0 || kb_total <= 0) return 0;
    static bool attr[MAXS + 1] = {false};
    const int bytes = S * SLOT + 2048;
    DenseArgs a;
    a.M = (int)M; a.N = (int)N;
    a.kb_total = kb_total;
    const int nsplit = dense_splits(M, N, kb_total, &a.kb_per_split);
    a.a_planes = A.planes; a.b_planes = B.planes;
    a.part = part;
    a.err = err;
    const dim3 grid((unsigned)((N + BN - 1) / BN), (unsigned)((M + BM - 1) / BM), (unsigned)nsplit);
#define HB_DENSE(SS)                                                                                    \
    do {                                                                                                \
        if (!attr[SS]) {                                                                                \
            cudaFuncSetAttribute(dense_split_kernel<SS>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes); \
            attr[SS] = true;                                                                            \
        }                                                                                               \
        dense_split_kernel<SS><<<grid, NTHREADS, bytes, s>>>(A.tm, B.tm, a);                            \
    } while (0)
    switch (S) {
        case 2: HB_DENSE(2); break;
        case 3: HB_DENSE(3); break;
        case 4: HB_DENSE(4); break;
        case 5: HB_DENSE(5); break;
        default: HB_DENSE(6); break;
    }
#undef HB_DENSE
    const int64_t tot = M * N;
    dense_reduce_kernel<<<(unsigned)((tot + 255) / 256), 256, 0, s>>>(part, nsplit, (int)M, (int)N, Y, ldy);
    return 2;
}

bool release_f64_slices(hb_ctx *ctx) {
    hb_ctx *owner = ctx->base ? ctx->base : ctx;
    if (!owner->mixed || !owner->mixed->panel[0].ready || *owner->batches > 0) return false;
    cudaDeviceSynchronize();
    for (hb_ctx *c : {ctx, owner})
        for (void **p : {&c->plan, &c->shard_plan})
            if (*p && plan_precision((Plan *)*p) == HB_FP64) {
                plan_destroy((Plan *)*p);
                *p = nullptr;
            }
    PanelSlices &PS = owner->mixed->panel[0];
    dfree(owner, PS.buf);
    dfree(owner, PS.scales);
    PS = PanelSlices();
    if (ctx != owner && ctx->mixed) ctx->mixed->panel[0] = PanelSlices();
    ++owner->tables_gen;          // other borrowing contexts let go of them before their next build
    return true;
}

void release_mixed(hb_ctx *ctx) {
    if (!ctx->mixed) return;
    for (PanelSlices &P : ctx->mixed->panel)
        if (!P.borrowed) {
            dfree(ctx, P.buf);
            dfree(ctx, P.scales);
        }
    if (!ctx->mixed->panel[1].borrowed) dfree(ctx, ctx->mixed->pdiag);
    delete ctx->mixed;
    ctx->mixed = nullptr;
}
