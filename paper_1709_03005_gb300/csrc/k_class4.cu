// K4: class 4, continuum x L2 (Eq. 5).
//
// For L2 function l and target group g:
//   H~[l][(g n j)] = sum_{m partners of l} c_mn <D_m + j|H|chi_l>
// The classified (m, l) pairs (D_m within a single substitution of chi_l, so
// the (N+1)-electron pair is within a double excitation) are the prototypes;
// each gives, for every continuum orbital j, one or two integrals of the form
// (ab|c j) (plus h_jt for a single excitation), all contiguous in j in the
// (tt|tc) class array, so the threads of a block read them coalesced.
// A block owns one L2 row and a tile of continuum orbitals (one per thread)
// and keeps a tile of target states in registers; the CI rows of a batch of
// partners are staged in shared memory.
//   plain build: prototype values and the rank-1 accumulation in FP64;
//   mixed build: everything in double-float on the FP32 pipes (the FP64 pipe
//   of this part is 64 times narrower): the integrals, h and the CI vectors are
//   kept as (hi, lo) float pairs, the prototype sums use double-float adds,
//   the products c * y are exact by FMA and the accumulation is TwoSum based
//   (about 44 significant bits); the state tile and the thread count follow
//   the group's state and continuum counts.
#include "hb_df.cuh"
#include "hb_tasks.cuh"

namespace hb {

namespace {

constexpr int kJ = 224;     // most threads of a block
constexpr int kBatch = 32;

// A staged pair, worked out once for all orbitals and states: of degree 2 the
// first elements of its direct and exchange rows of the (tt|tc) table, of degree
// 1 (chi = D + t, the single excitation t -> j) the orbital t.
struct PairRec {
    int64_t dir, exc;      // -1: no such integral
    int col, t;            // the determinant; t >= 0: degree 1
    int neg, pad;
};

template <int W>
__device__ __forceinline__ PairRec pair_rec(const C4Task &T, const hb_pair &r) {
    const int sb = 64 * W, n_to = T.I.n_to, cont_spin = T.cont_spin;
    PairRec p;
    p.dir = p.exc = -1;
    p.col = r.col;
    p.t = -1;
    p.neg = r.phase < 0;
    p.pad = 0;
    if (r.degree == 1) {
        p.t = r.hole[0] % sb;
        return p;
    }
    // degree 2: holes h1 < h2 in chi, particles {q, continuum} in D + j
    const int h1 = r.hole[0], h2 = r.hole[1], q = r.part[0];
    const int kq = 2 * q, kv = cont_spin == 0 ? 2 * 64 * W - 1 : 2 * 128 * W - 1;
    const int s1 = h1 / sb, s2 = h2 / sb, sq = q / sb;
    const int o1 = h1 % sb, o2 = h2 % sb, oq = q % sb;
    // (q h1|j h2) and (q h2|j h1)
    const int64_t x12 = (pair_idx(oq, o1) * n_to + o2) * T.I.n_co, x21 = (pair_idx(oq, o2) * n_to + o1) * T.I.n_co;
    if (kq < kv) {
        if (sq == s1 && cont_spin == s2) p.dir = x12;
        if (sq == s2 && cont_spin == s1) p.exc = x21;
    } else {
        // the continuum orbital is the first particle
        if (cont_spin == s1 && sq == s2) p.dir = x21;
        if (cont_spin == s2 && sq == s1) p.exc = x12;
    }
    return p;
}

// The integrals of a task, FP64 or as float pairs (Acc of hb_df.cuh), for
// continuum orbital j.
template <int W, class Acc>
struct Prototype {
    const double *x, *h;
    const float2 *x_df, *h_df;
    int64_t plane;
    int n_co, cont_spin;
    typename Acc::Entry dir, exc;
    __device__ __forceinline__ Prototype(const C4Task &T, int j)
        : x(T.I.tttc + j), h(T.I.h + (int64_t)(T.I.n_to + j) * T.I.n_orb), x_df(T.tttc_df + j),
          h_df(T.h_df + (int64_t)(T.I.n_to + j) * T.I.n_orb), plane((int64_t)T.I.n_to * T.I.n_co), n_co(T.I.n_co),
          cont_spin(T.cont_spin) {}
    // starts the reads of a pair of degree 2
    __device__ __forceinline__ void fetch(const PairRec &p) {
        dir = exc = typename Acc::Entry{};
        if (p.dir >= 0) dir = Acc::entry(x, x_df, p.dir);
        if (p.exc >= 0) exc = Acc::entry(x, x_df, p.exc);
    }
    // <D_m + j|H|chi_l> without its sign; of degree 2 from what fetch read
    __device__ __forceinline__ Acc value(const PairRec &p, const uint64_t *__restrict__ dets) const {
        Acc v;
        if (p.t < 0) {
            v.add_entry(dir);
            v.sub_entry(exc);
            return v;
        }
        const uint64_t *D = dets + (int64_t)p.col * 2 * W;
        const int t = p.t;
        v.add(h, h_df, t);
#pragma unroll
        for (int w = 0; w < 2 * W; ++w) {
            uint64_t y = __ldg(D + w);
            const int s = w / W;
            while (y) {
                const int k = 64 * (w % W) + __ffsll((long long)y) - 1;
                y &= y - 1;
                v.add(x, x_df, pair_idx(k, k) * plane + (int64_t)t * n_co);                         // (jt|kk)
                if (s == cont_spin) v.sub(x, x_df, pair_idx(k, t) * plane + (int64_t)k * n_co);     // (jk|kt)
            }
        }
        return v;
    }
};

// Block = blockDim.x continuum orbitals of one L2 row; NS target states per
// pass.  FP64 FMAs for states beyond the group's cost as much as the others on
// this pipe: with one tile of 32 states and 128 threads, 20 states x 150
// orbitals took 1.19 ms and 7 x 37 0.16 ms, now 0.53 and 0.05.
template <int W, int NS>
__global__ void __launch_bounds__(kJ)
class4_kernel(const C4Task *__restrict__ tasks, const int64_t *__restrict__ blk, int n_tasks) {
    __shared__ double cs[kBatch][NS];
    __shared__ PairRec rs[kBatch];
    const int ti = task_of(blk, n_tasks, blockIdx.x);
    const C4Task &T = tasks[ti];
    const int JT = blockDim.x;
    const hb_pair *__restrict__ pairs = T.pairs;
    const uint64_t *__restrict__ dets = T.dets;
    const double *__restrict__ C = T.C;
    const int ns = T.ns, cf = T.cf, cn = T.cn;
    const int lb = (int)(blockIdx.x - blk[ti]);
    const int l = lb / T.ny;
    const int jl = (lb % T.ny) * JT + threadIdx.x;
    const bool jv = jl < cn, wv = jl - (int)(threadIdx.x & 31) < cn;   // this lane's, this warp's orbitals exist
    Prototype<W, AccD> proto(T, cf + (jv ? jl : 0));
    const int64_t b = T.row_ptr[l], e = T.row_ptr[l + 1];
    for (int n0 = 0; n0 < ns; n0 += NS) {
        const int nc = min(NS, ns - n0);
        double acc[NS];
#pragma unroll
        for (int n = 0; n < NS; ++n) acc[n] = 0.0;
        for (int64_t p0 = b; p0 < e; p0 += kBatch) {
            const int cnt = (int)(e - p0 < kBatch ? e - p0 : kBatch);
            __syncthreads();
            for (int t = threadIdx.x; t < cnt; t += JT) rs[t] = pair_rec<W>(T, pairs[p0 + t]);
            __syncthreads();
            for (int t = threadIdx.x; t < cnt * NS; t += JT) {
                const int i = t / NS, n = t % NS;
                cs[i][n] = n < nc ? C[(int64_t)rs[i].col * ns + n0 + n] : 0.0;
            }
            __syncthreads();
            proto.fetch(rs[0]);
            for (int i = 0; i < (wv ? cnt : 0); ++i) {
                AccD v = proto.value(rs[i], dets);
                if (rs[i].neg) v.neg();
                const double y = v.v;
                if (i + 1 < cnt) proto.fetch(rs[i + 1]);     // in flight during the sums
#pragma unroll
                for (int n = 0; n < NS; ++n) acc[n] = fma(cs[i][n], y, acc[n]);
            }
        }
        if (jv) {
            double *out = T.Hlc + (int64_t)l * T.ld + T.col_off + jl;
#pragma unroll
            for (int n = 0; n < NS; ++n)
                if (n < nc) out[(int64_t)(n0 + n) * cn] = acc[n];
        }
    }
}

// ------------------------------------------------------- double-float path
// Block = blockDim.x continuum orbitals of one L2 row; NS
// target states per pass, two to an f32x2 instruction.  The CI coefficients lie
// in shared memory as high and low words, four states to a load.
// Issue and latency bind it: 5000 rows, 150 orbitals, 20 states, 74000 pairs took
// 0.28 ms when every thread decoded every pair (500 instructions a pair and warp)
// in blocks of 32 orbitals that each staged the same rows, now 0.21.
template <int W, int NS>
__global__ void __launch_bounds__(kJ, NS <= 24 ? 3 : 1)
class4_df_kernel(const C4Task *__restrict__ tasks, const int64_t *__restrict__ blk, int n_tasks) {
    static_assert(NS % 4 == 0, "coefficients are read four states at a time");
    __shared__ __align__(16) float ch[kBatch][NS], cl[kBatch][NS];
    __shared__ PairRec rs[kBatch];
    const int ti = task_of(blk, n_tasks, blockIdx.x);
    const C4Task &T = tasks[ti];
    const int JT = blockDim.x;
    const int ns = T.ns, cn = T.cn;
    const int lb = (int)(blockIdx.x - blk[ti]);
    const int l = lb / T.ny;
    const int jl = (lb % T.ny) * JT + threadIdx.x;
    const bool jv = jl < cn, wv = jl - (int)(threadIdx.x & 31) < cn;   // this lane's, this warp's orbitals exist
    Prototype<W, AccF> proto(T, T.cf + (jv ? jl : 0));
    const uint64_t *__restrict__ dets = T.dets;
    const int64_t b = T.row_ptr[l], e = T.row_ptr[l + 1];
    for (int n0 = 0; n0 < ns; n0 += NS) {
        const int nc = min(NS, ns - n0);
        f2 ahi[NS / 2], alo[NS / 2];
#pragma unroll
        for (int n = 0; n < NS / 2; ++n) { ahi[n] = f2_pack(0.0f, 0.0f); alo[n] = f2_pack(0.0f, 0.0f); }
        for (int64_t p0 = b; p0 < e; p0 += kBatch) {
            const int cnt = (int)(e - p0 < kBatch ? e - p0 : kBatch);
            __syncthreads();
            for (int t = threadIdx.x; t < cnt; t += JT) rs[t] = pair_rec<W>(T, T.pairs[p0 + t]);
            __syncthreads();
            for (int t = threadIdx.x; t < cnt * NS; t += JT) {
                const int i = t / NS, n = t % NS;
                const float2 c = n < nc ? __ldg(T.C_df + (int64_t)rs[i].col * ns + n0 + n) : make_float2(0.0f, 0.0f);
                ch[i][n] = c.x;
                cl[i][n] = c.y;
            }
            __syncthreads();
            proto.fetch(rs[0]);
            for (int i = 0; i < (wv ? cnt : 0); ++i) {
                AccF v = proto.value(rs[i], dets);
                if (rs[i].neg) v.neg();
                const f2 y = f2_pack(v.h, v.h), ny = f2_pack(-v.h, -v.h), yl2 = f2_pack(v.l, v.l);
                if (i + 1 < cnt) proto.fetch(rs[i + 1]);     // in flight during the sums
#pragma unroll
                for (int n = 0; n < NS; n += 4) {
                    const ulonglong2 h4 = *reinterpret_cast<const ulonglong2 *>(&ch[i][n]);
                    const ulonglong2 l4 = *reinterpret_cast<const ulonglong2 *>(&cl[i][n]);
                    df_fma(ahi[n / 2], alo[n / 2], y, ny, yl2, f2{h4.x}, f2{l4.x});
                    df_fma(ahi[n / 2 + 1], alo[n / 2 + 1], y, ny, yl2, f2{h4.y}, f2{l4.y});
                }
            }
            // renormalise once per batch so the low words stay small
#pragma unroll
            for (int n = 0; n < NS / 2; ++n) df_norm(ahi[n], alo[n]);
        }
        if (jv) {
            double *out = T.Hlc + (int64_t)l * T.ld + T.col_off + jl;
#pragma unroll
            for (int n = 0; n < NS; n += 2) {
                float h0, h1, l0, l1;
                f2_unpack(ahi[n / 2], h0, h1);
                f2_unpack(alo[n / 2], l0, l1);
                if (n < nc) out[(int64_t)(n0 + n) * cn] = df_sum(h0, l0);
                if (n + 1 < nc) out[(int64_t)(n0 + n + 1) * cn] = df_sum(h1, l1);
            }
        }
    }
}

__global__ void split_df_kernel(const double *__restrict__ x, int64_t n, float2 *__restrict__ out) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double v = x[i];
    const float h = (float)v;
    out[i] = make_float2(h, (float)(v - (double)h));
}

}  // namespace

int class4_ny(int cn, int jt) { return (cn + jt - 1) / jt; }
int64_t blocks_class4(int n_l2, int cn, int jt) { return cn > 0 ? (int64_t)n_l2 * class4_ny(cn, jt) : 0; }

// State tile and thread count of either kernel for a group (host side):
// the fewest passes over the states, then the smallest tile; the continuum
// tile that leaves the fewest idle threads (ties to the larger block).
void class4_shape(int ns, int cn, int *ns_tile, int *jt) {
    // passes of at most 32 states (larger tiles cost more in registers and
    // occupancy than the prototype values recomputed per pass), the state
    // tile rounded up to a multiple of 4 (8 beyond 32)
    const int passes = (ns + 31) / 32;
    const int need = (ns + passes - 1) / passes;
    *ns_tile = need <= 4 ? 4 : (need + 3) / 4 * 4;
    // one block for the whole row where the orbitals allow it (the pairs and CI
    // rows are staged once), else blocks of one size
    const int tiles = (cn + kJ - 1) / kJ, per = tiles > 0 ? (cn + tiles - 1) / tiles : 1;
    *jt = (per + 31) / 32 * 32;
}

void split_df(const double *x, int64_t n, float2 *out, cudaStream_t s) {
    if (n <= 0) return;
    split_df_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(x, n, out);
}

int g_class4(const Grouped<C4Task> &g, int W, int dfloat, int ns_tile, int jt, cudaStream_t s) {
    if (g.blocks <= 0) return 0;
    const unsigned grid = (unsigned)g.blocks;
#define HB_C4(WW)                                                                          \
    switch (ns_tile) {                                                                     \
        case 4: class4_kernel<WW, 4><<<grid, jt, 0, s>>>(g.tasks, g.blk, g.n); break;      \
        case 8: class4_kernel<WW, 8><<<grid, jt, 0, s>>>(g.tasks, g.blk, g.n); break;      \
        case 12: class4_kernel<WW, 12><<<grid, jt, 0, s>>>(g.tasks, g.blk, g.n); break;    \
        case 16: class4_kernel<WW, 16><<<grid, jt, 0, s>>>(g.tasks, g.blk, g.n); break;    \
        case 20: class4_kernel<WW, 20><<<grid, jt, 0, s>>>(g.tasks, g.blk, g.n); break;    \
        case 24: class4_kernel<WW, 24><<<grid, jt, 0, s>>>(g.tasks, g.blk, g.n); break;    \
        case 28: class4_kernel<WW, 28><<<grid, jt, 0, s>>>(g.tasks, g.blk, g.n); break;    \
        default: class4_kernel<WW, 32><<<grid, jt, 0, s>>>(g.tasks, g.blk, g.n); break;    \
    }
    if (!dfloat) {
        switch (W) {
            case 1: HB_C4(1); break;
            case 2: HB_C4(2); break;
            case 3: HB_C4(3); break;
            default: HB_C4(4); break;
        }
#undef HB_C4
        return 1;
    }
#define HB_C4DF(WW)                                                                                       \
    switch (ns_tile) {                                                                                    \
        case 4: class4_df_kernel<WW, 4><<<grid, jt, 0, s>>>(g.tasks, g.blk, g.n); break;                 \
        case 8: class4_df_kernel<WW, 8><<<grid, jt, 0, s>>>(g.tasks, g.blk, g.n); break;                 \
        case 12: class4_df_kernel<WW, 12><<<grid, jt, 0, s>>>(g.tasks, g.blk, g.n); break;               \
        case 16: class4_df_kernel<WW, 16><<<grid, jt, 0, s>>>(g.tasks, g.blk, g.n); break;               \
        case 20: class4_df_kernel<WW, 20><<<grid, jt, 0, s>>>(g.tasks, g.blk, g.n); break;               \
        case 24: class4_df_kernel<WW, 24><<<grid, jt, 0, s>>>(g.tasks, g.blk, g.n); break;               \
        case 28: class4_df_kernel<WW, 28><<<grid, jt, 0, s>>>(g.tasks, g.blk, g.n); break;               \
        case 32: class4_df_kernel<WW, 32><<<grid, jt, 0, s>>>(g.tasks, g.blk, g.n); break;               \
        case 40: class4_df_kernel<WW, 40><<<grid, jt, 0, s>>>(g.tasks, g.blk, g.n); break;               \
        case 48: class4_df_kernel<WW, 48><<<grid, jt, 0, s>>>(g.tasks, g.blk, g.n); break;               \
        case 56: class4_df_kernel<WW, 56><<<grid, jt, 0, s>>>(g.tasks, g.blk, g.n); break;               \
        default: class4_df_kernel<WW, 64><<<grid, jt, 0, s>>>(g.tasks, g.blk, g.n); break;               \
    }
    switch (W) {
        case 1: HB_C4DF(1); break;
        case 2: HB_C4DF(2); break;
        case 3: HB_C4DF(3); break;
        default: HB_C4DF(4); break;
    }
#undef HB_C4DF
    return 1;
}

}  // namespace hb
