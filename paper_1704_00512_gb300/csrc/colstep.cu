// The recursion in column order on the tensor cores: several steps of the
// masked Chebyshev recursion (Eq. 3) per launch, fused with the accumulation
// of several expansions (Eq. 1) and the moments Tr T_k, <T_k, G>.
//
// Column J of T_{k+1} needs only column J of T_k and T_{k-1} (Sec. "Expansion
// in Chebyshev polynomials"), so a panel of P neighbouring block columns (4 in
// FP32 / BF16, 2 in FP64) runs through all the steps of a launch in one thread
// block, with no data from any other.  T_k is kept in *column order*: the
// blocks (K, J) of column J are contiguous, at the BCSR positions of row J of
// the symmetric output pattern; two buffers, T_{k+1} over T_{k-1}.
//
// What bounds it.  The products are gathered 4x4 blocks.  On the FMA pipes
// they cost 64 instructions a block and panel column (FP64 at 1/64 of the FP32
// rate; FP32 bound by issue and by shared-memory reads, 240 instructions per
// 16 entries).  Here they are f16 tensor-core products of *digits*: within a
// panel column (and within a scalar row of the operator) every value is written on
// one power-of-two grid as a sum of small integers times powers of two, three
// digits (30 bits) for FP32 and six (60 bits) for FP64.  Integers up to 2048
// are exact in f16, and the products of one mma are small enough for the FP32
// accumulators to hold the leading digit sums D_s = sum_{i+j=s} d_i d_j exactly:
//     FP32: D_0 exact (below 2^24 over two mma, then added to an FP32 sum, round
//           to nearest), D_1, D_2 (weights 2^-10, 2^-20) kept in the accumulator; 6 mma
//           per 16 operator rows, 16 inner and 8 panel columns;
//     FP64: D_0 .. D_3 exact (summed as integers), D_4 .. D_6 (weights 2^-40,
//           2^-50, 2^-60) in two accumulators; 26 mma.
// Exactness matters beyond the size of the rounding: a tensor core that
// truncates its sums would shrink every product by about 2^-25, the same way
// at every step, which acts like a scaled operator.  What is left are the grids
// themselves (an element counts to 2^-30 or 2^-60 of the largest of its column of T_k or
// its scalar row of the operator) and the terms beyond the last digit sum.  Error of 64-term expansions of 140 and 150 atoms
// against long doubles, largest of the accumulators, before -> now: FP64 Fermi 3.5e-16
// -> 3.5e-16, powers 9.4e-16 -> 5.3e-16 (without D_6 3.7e-16 and 1.0e-15); FP32
// Fermi 3.5e-8 -> 2.9e-8, powers 4.7e-7 -> 2.5e-7; FP64-accurate 4.2e-14 -> 5.3e-16.
// Measured (GB300): one step at 1,500 atoms, r_c 10, r_out 14 bohr, three
// accumulators: FP64 9.2 -> 1.3 ms, FP64-accurate (before: double-floats) at 1,000
// atoms, 8 / 12 bohr: 2.3 -> 0.35 ms; FP32 at 10,000 atoms 3.47 -> 2.65 ms, at 1,000
// atoms, 8 / 12 bohr: 0.237 -> 0.128 ms, at 3,000 atoms with four functions 1.12 ->
// 0.87 ms.  ncu: L1 access cycles 65 % (FP64) and 58 % (FP32), ALU (digit unpacking) 44 %
// and 50 %, tensor pipe 48 % and 37 %: an operator block of 64 or 128 bytes is used for
// one row group and panel only, and an L1 load costs a cycle per line that the lanes it
// serves together touch.
// Tried without gain: f16 operator digits in memory (96 bytes: 3.7 instead of 2.9 ms
// at 10,000 atoms), 12 warps (10 % slower), lanes over two blocks per access (L1
// cycles -35 %, instructions +30 %, 15 % slower).
//
// One thread block per panel.  Per step:
//   1. the panel's T_k blocks become digits in shared memory, X[slot][column]
//      (slot = rank of the block row in the union of the columns' row lists);
//      the grid of each column comes from the largest element that the step
//      before wrote;
//   2. each warp takes groups of 4 union rows.  The operator blocks of the
//      group with K in the union are listed by merged K, four slots ("quad") at
//      a time: an m16n8k16 product of the operator's 16 rows (A, from the
//      operator's digits in L2) with 8 panel columns (B, from X); rows without
//      a block at a merged K name a zero block;
//   3. at the end of a group each lane holds 2 neighbouring elements of the
//      blocks (row, column) and finishes them: T_{k+1} = 2 M~ T_k - T_{k-1}, and
//      every third step acc_j += c_j T of the last three terms (in the order of
//      one term per step) and their parts of the moments;
//   4. the panel's moments go to a table that a second kernel sums in a fixed
//      order.
// Elements that are not finite spread by a pass of their own (mark_not_finite).  A column
// beyond the grid's exponents, or an operator with such elements or ones that are not
// finite, takes the step in plain FP32 / FP64 instead (slow: 1.7 ms a step at 1,000 atoms
// in FP32, 0.12 by digits).  An expansion that leaves its interval stays on the digits to
// the end of the finite numbers and beyond: 800 terms there with bounds 5 % too narrow,
// overflowing at term 279, take 120 ms (96 in bounds; 985 when every column that was not
// finite sent its panel to the plain products, 178 on the FMA pipe).
#include <algorithm>
#include <array>
#include <numeric>
#include <thread>

#include "common.cuh"
#include "digits.cuh"
#include "kernels.cuh"
#include "plan.cuh"

namespace cheb {

struct ColArgs {
    const int32_t *panels;  // (first column, column count, union rows, system) per panel
    const int32_t *order;   // panel of each thread block
    const int32_t *wchunk;  // [panels][NW + 1] quad range of each warp
    const int32_t *wrow;    // [panels][NW + 1] group range of each warp
    const uint32_t *rows;   // per group: the 4 union slots and the quad count (2 words)
    const uint32_t *ent;    // [quads][16] operator block << COL_SLOT_BITS | union slot
    const uint16_t *slot;   // union slot of each column-order block
    const int64_t *rp;      // P_out row_ptr = column starts in column order
    const int32_t *ci;      // row of each column-order block
    const int32_t *tperm;   // BCSR position of each column-order block
    const int64_t *Lrp;     // operator pattern and FP64 values
    const int32_t *Lci;
    const double *Lv;
    int64_t nnzL;
    const uint4 *opd;       // operator digits (one zero block appended)
    const int32_t *opexp;   // grid exponents of the operator's scalar rows
    const int32_t *opflag;  // nonzero: an operator element beyond the digits
    void *T[2];             // T_k in T[k & 1] (column order)
    int32_t t0, t1;         // terms formed by this launch: t0 .. t1 - 1 (t0 = 2: also terms 0 and 1)
    const int32_t *n_terms;  // per system, or NULL: n_single
    int32_t n_single;
    int32_t nf;
    double *acc[MAX_F];   // the caller's FP64 accumulators (BCSR order)
    float *accp[MAX_F];   // FP32: the accumulators as (hi, lo) float pairs, column order
    const double *coef;   // coef[coef_off[sys] + f * coef_stride + k]
    const int64_t *coef_off;
    int32_t coef_stride;
    const double *G;      // the caller's G (BCSR order) or NULL
    float *Gp;            // FP32: G as (hi, lo) float pairs in column order
    double *part;         // [panel][pstride][2] moments of terms tbase ..
    int32_t pstride, tbase, want_mom;
    int32_t round_bf16;
};

// Double-float arithmetic (a value is an unevaluated sum hi + lo of two
// floats, about 48 significant bits): GB300 issues FP64 at 1/64 of the FP32
// rate, so the per-step FP64 accumulation of Eq. 1 and the trace functional
// are carried on the FP32 pipe with error-free transformations (Knuth's
// two-sum, the FMA product error) and converted to FP64 once per expansion.
__device__ __forceinline__ void ff_add_prod(float &hi, float &lo, float y, float ch, float cl) {
    // (hi, lo) += y * (ch + cl)
    const float p = __fmul_rn(y, ch);
    float pe = __fmaf_rn(y, ch, -p);
    pe = __fmaf_rn(y, cl, pe);
    const float s = __fadd_rn(hi, p);
    const float bb = __fsub_rn(s, hi);
    const float e = __fadd_rn(__fsub_rn(hi, __fsub_rn(s, bb)), __fsub_rn(p, bb));
    const float t = __fadd_rn(__fadd_rn(lo, pe), e);
    hi = __fadd_rn(s, t);
    lo = __fsub_rn(t, __fsub_rn(hi, s));
}
__host__ __device__ inline void ff_split(double v, float &hi, float &lo) {
    hi = (float)v;
    lo = (float)(v - (double)hi);
}


template <typename T>
struct Vec2;
template <>
struct Vec2<float> {
    using V = float2;
};
template <>
struct Vec2<double> {
    using V = double2;
};

// The products of one group in plain FP32 / FP64, from the FP64 operator and T_k
// (R): out[4 j + 2 h + c] for tile j, row half h, column 2t + c, where the mma has
// them.
template <typename T>
__device__ __noinline__ void plain_group(const ColArgs &a, const int32_t *opos, const T *R, const uint32_t *ent, int cnt,
                                         int lane, T *out) {
    constexpr int NT = Dig<T>::NT, P = 2 * NT;
    const int g = lane >> 2, t = lane & 3;
    for (int i = 0; i < 4 * NT; ++i) out[i] = T(0);
    for (int e = 0; e < 8 * cnt; ++e) {  // quad e / 8, slot (e / 2) % 4, row half e % 2
        const uint32_t w = ent[(e >> 3) * COL_CW + ((g >> 2) * 4 + ((e >> 1) & 3)) * 2 + (e & 1)];
        const uint32_t blk = w >> COL_SLOT_BITS, sl = w & ((1u << COL_SLOT_BITS) - 1u);
        if (blk == (uint32_t)a.nnzL) continue;
        for (int m = 0; m < 4; ++m) {
            T hv = (T)a.Lv[(int64_t)blk * BB + 4 * (g & 3) + m];
            if constexpr (sizeof(T) == 4) {
                if (a.round_bf16) hv = bf16r(hv);
            }
            for (int j = 0; j < NT; ++j) {
                const int p = opos[sl * P + 2 * j + (t >> 1)];
                if (p < 0) continue;
                const T *x = R + (int64_t)p * BB + 4 * m + 2 * (t & 1);
                T *o = out + 4 * j + 2 * (e & 1);
                o[0] = mac(hv, __ldcg(x), o[0]);
                o[1] = mac(hv, __ldcg(x + 1), o[1]);
            }
        }
    }
}

// Before a step of a panel with elements of T_{term-1} (R) that are not finite: the largest
// finite elements of its columns (into mx), and NaN in T_{term-2} (C) wherever a product
// with one of the others goes.  T_term is then NaN there by its own sum, and the digits of
// the finite elements do the rest: an expansion that leaves its interval, whose columns
// overflow one after the other, goes on at the others' speed.  nf: the columns of each
// union row's blocks with such an element, 16 bits.
template <typename T>
__device__ __noinline__ void mark_not_finite(const ColArgs &a, int par, uint32_t *mx) {
    extern __shared__ __align__(16) unsigned char smem[];
    constexpr int NT = Dig<T>::NT, P = 2 * NT, NC = 8 * NT, NTH = COL_NW * 32;
    constexpr uint32_t SM = (1u << COL_SLOT_BITS) - 1u;
    constexpr ColLayout lay = col_layout(P);
    const int32_t *opos = reinterpret_cast<const int32_t *>(smem + lay.off_pos);
    const uint2 *srow = reinterpret_cast<const uint2 *>(smem + lay.off_rows);
    uint32_t *nf = reinterpret_cast<uint32_t *>(smem + lay.off_nf);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int pid = a.order[blockIdx.x], nu = a.panels[4 * pid + 2];
    const int32_t *wr = a.wrow + pid * (COL_NW + 1);
    const T *R = static_cast<const T *>(a.T[par ^ 1]);
    T *C = static_cast<T *>(a.T[par]);
    __syncthreads();  // (every thread has read mx)
    if (tid < NC) mx[tid] = 0u;
    for (int i = tid; i < (nu + 1) / 2; i += NTH) nf[i] = 0u;
    __syncthreads();
    for (int i = tid; i < nu * P; i += NTH) {
        const int p = opos[i], s = i / P, q = i % P;
        if (p < 0) continue;
        for (int e = 0; e < 16; ++e) {
            const uint32_t m = mag_bits(__ldcg(R + (int64_t)p * BB + e));
            const int c = 4 * q + (e & 3);
            if (m >= NOT_FINITE<T>) atomicOr(&nf[s >> 1], (1u << c) << (16 * (s & 1)));
            else if (m > mx[c]) atomicMax(&mx[c], m);
        }
    }
    __syncthreads();
    // the warp's groups: a lane has word (lane % 16) of every second quad, of row a
    const int a4 = ((lane >> 3) & 1) | ((lane & 1) << 1);
    const uint32_t *ent = a.ent + (int64_t)a.wchunk[pid * (COL_NW + 1) + warp] * COL_CW;
    for (int r = wr[warp] - wr[0]; r < wr[warp + 1] - wr[0]; ++r) {
        const uint2 rw = srow[r];
        const int cnt = (int)(rw.y >> COL_SLOT_BITS);
        uint32_t bits = 0u;
        for (int k = lane; k < cnt * COL_CW; k += 32) {
            const uint32_t w = __ldg(ent + k), s = w & SM;
            if ((w >> COL_SLOT_BITS) != (uint32_t)a.nnzL) bits |= nf[s >> 1] >> (16 * (s & 1)) & 0xffffu;
        }
        ent += cnt * COL_CW;
        for (int o = 2; o < 32; o = o == 4 ? 16 : 2 * o) bits |= __shfl_xor_sync(0xffffffffu, bits, o);
        const uint32_t s = a4 == 3 ? rw.y & SM : (rw.x >> (a4 * COL_SLOT_BITS)) & SM;
        // (the lanes of a row share its columns)
        for (int q = 0; q < P && s != SM; ++q) {
            const int p = opos[s * P + q], c = (lane >> 1) & 3;
            if (p >= 0 && lane < 16 && (bits >> (4 * q + c)) & 1u)
                for (int e = 0; e < 4; ++e) C[(int64_t)p * BB + 4 * e + c] = T(NAN);
        }
    }
    // (the barrier before the products orders these stores before their loads)
}

template <typename T>
__global__ void __launch_bounds__(COL_NW * 32, 1) k_colstep(const __grid_constant__ ColArgs a) {
    using D = Dig<T>;
    using V2 = typename Vec2<T>::V;
    constexpr int NT = D::NT, P = 2 * NT, NTH = COL_NW * 32, NC = 8 * NT;
    constexpr bool F64 = sizeof(T) == 8;
    constexpr ColLayout lay = col_layout(P);
    constexpr int XV = lay.slot_bytes / 16;  // 16-byte chunks of a slot's digits
    constexpr uint32_t SM = (1u << COL_SLOT_BITS) - 1u;
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ uint32_t s_max[2][NC];
    __shared__ int s_e[NC];
    __shared__ float s_cf[NC];  // FP32: 2^(e - 1)
    __shared__ int s_slow, s_marked;  // (shared, so that no register holds them)
    __shared__ int s_cb[P + 1];
    __shared__ int s_dslot[P];
    __shared__ float s_ch[3][MAX_F], s_cl[3][MAX_F];
    __shared__ double s_c[3][MAX_F];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int pid = a.order[blockIdx.x];
    const int j0 = a.panels[4 * pid], nc = a.panels[4 * pid + 1], nu = a.panels[4 * pid + 2], sys = a.panels[4 * pid + 3];
    const int n = a.n_terms ? a.n_terms[sys] : a.n_single;
    if (a.t0 >= n && a.t0 != 2) return;  // this system is done
    uint4 *X = reinterpret_cast<uint4 *>(smem + lay.off_x);
    uint32_t *X2 = reinterpret_cast<uint32_t *>(smem + lay.off_x + 256);  // FP32: the third digits, behind the others
    int32_t *opos = reinterpret_cast<int32_t *>(smem + lay.off_pos);
    int8_t *rexp = reinterpret_cast<int8_t *>(smem + lay.off_rexp);  // of the union rows' scalar rows
    uint2 *srow = reinterpret_cast<uint2 *>(smem + lay.off_rows);
    double *red = reinterpret_cast<double *>(smem + lay.off_red);
    const double *coef = a.coef ? a.coef + (a.coef_off ? a.coef_off[sys] : 0) : nullptr;
    double *part = a.part + (int64_t)pid * a.pstride * 2;

    // --- the panel: column starts, block positions, zero digits
    if (tid <= P) s_cb[tid] = (int)a.rp[j0 + min(tid, nc)];
    if (tid < P) s_dslot[tid] = -1;
    if (tid == 0) s_marked = 0;
    if (tid < 2 * NC) (&s_max[0][0])[tid] = 0u;
    for (int i = tid; i < nu * XV; i += NTH) {
        const uint32_t z = !F64 && i % XV >= 16 ? 0x80808080u : 0u;
        X[i] = make_uint4(z, z, z, z);
    }
    for (int i = tid; i < nu * P; i += NTH) opos[i] = -1;
    const int rbase = a.wrow[pid * (COL_NW + 1)];  // the panel's first group
    for (int i = tid; i < (nu + 3) / 4; i += NTH) srow[i] = reinterpret_cast<const uint2 *>(a.rows)[rbase + i];
    __syncthreads();
    const int cb0 = s_cb[0], cb1 = s_cb[nc];  // (block indexes fit 31 bits)
    auto col_of = [&](int b) {
        int q = 0;
#pragma unroll
        for (int qq = 1; qq < P; ++qq)
            if (qq < nc && b >= s_cb[qq]) q = qq;
        return q;
    };
    for (int b = cb0 + tid; b < cb1; b += NTH) {
        const int q = col_of(b), s = a.slot[b], K = a.ci[b];
        opos[s * P + q] = (int32_t)b;
        const int4 e = *reinterpret_cast<const int4 *>(a.opexp + 4 * K);
        *reinterpret_cast<char4 *>(rexp + 4 * s) = make_char4(e.x, e.y, e.z, e.w);
        if (K == j0 + q) s_dslot[q] = s;
    }

    // block-wide sums of NV values to dst[0..NV-1] in a fixed order
    auto reduce_to = [&](auto &v, auto NVc, auto store) {
        constexpr int NV = decltype(NVc)::value;
#pragma unroll
        for (int i = 0; i < NV; ++i) {
            const double w = warp_sum(v[i]);
            if (lane == 0) red[warp * NV + i] = w;
        }
        __syncthreads();
        if (tid < NV) {
            double s = 0.0;
            for (int w = 0; w < COL_NW; ++w) s += red[w * NV + tid];
            store(tid, s);
        }
        __syncthreads();
    };

    // --- terms 0 and 1: T_0 = I, T_1 = M~, accumulators c_0/2 T_0 + c_1 T_1
    T *const Tb[2] = {static_cast<T *>(a.T[0]), static_cast<T *>(a.T[1])};
    if (a.t0 == 2) {
        double mv[4] = {0.0, 0.0, 0.0, 0.0};  // Tr T_0, <T_0, G>, Tr T_1, <T_1, G>
        for (int b = cb0 + tid; b < cb1; b += NTH) {
            const int J = j0 + col_of(b), K = a.ci[b];
            const int64_t la = find_in_row(a.Lrp, a.Lci, K, J);
            const int64_t o = (int64_t)a.tperm[b] * BB;
#pragma unroll 4
            for (int i = 0; i < 16; ++i) {
                const bool dg = K == J && (i % 5) == 0;
                const T v0 = dg ? T(1) : T(0);
                T v1 = la >= 0 ? (T)a.Lv[la * BB + i] : T(0);
                if constexpr (!F64) {
                    if (a.round_bf16) v1 = bf16r(v1);
                }
                Tb[0][(int64_t)b * BB + i] = v0;
                Tb[1][(int64_t)b * BB + i] = v1;
                const double d0 = (double)v0, d1 = (double)v1;
                for (int f = 0; f < a.nf; ++f) {
                    const double *cf = coef + (int64_t)f * a.coef_stride;
                    const double w = 0.5 * __ldg(cf) * d0 + __ldg(cf + 1) * d1;
                    if constexpr (F64) a.acc[f][o + i] = w;
                    else {
                        float hi, lo;
                        ff_split(w, hi, lo);
                        *reinterpret_cast<float2 *>(a.accp[f] + ((int64_t)b * BB + i) * 2) = make_float2(hi, lo);
                    }
                }
                if (a.G) {
                    const double gval = a.G[o + i];
                    mv[1] += gval * d0;
                    mv[3] += gval * d1;
                    if constexpr (!F64) {
                        float hi, lo;
                        ff_split(gval, hi, lo);
                        *reinterpret_cast<float2 *>(a.Gp + ((int64_t)b * BB + i) * 2) = make_float2(hi, lo);
                    }
                }
                if (dg) {
                    mv[0] += d0;
                    mv[2] += d1;
                }
            }
        }
        if (a.want_mom) reduce_to(mv, std::integral_constant<int, 4>(), [&](int i, double s) { part[i] = s; });
    }
    __syncthreads();
    const int tend = min(a.t1, n);
    // largest elements of the columns of T_{t0 - 1}
    if (a.t0 < tend) {
        const T *R = Tb[(a.t0 - 1) & 1];
        for (int b = cb0 + tid; b < cb1; b += NTH) {
            const int q = col_of(b);
            uint32_t m[4] = {0u, 0u, 0u, 0u};
#pragma unroll
            for (int i = 0; i < 16; ++i) m[i & 3] = max(m[i & 3], mag_bits(R[(int64_t)b * BB + i]));
#pragma unroll
            for (int c = 0; c < 4; ++c) atomicMax(&s_max[a.t0 & 1][4 * q + c], m[c]);
        }
        __syncthreads();
    }

    const int g = lane >> 2, t = lane & 3;  // mma row / column lane, slot of the quad
    const bool opbad = *a.opflag != 0;

    for (int term = a.t0; term < tend; ++term) {
        const int par = term & 1;
        const T *R = Tb[par ^ 1];  // T_{term-1}
        T *C = Tb[par];            // T_{term-2}, replaced by T_term
        // terms accumulated by this step: bit i of grp is term - i
        int grp = 0;
        if (term == n - 1 || (term >= 4 && (term - 1) % 3 == 0)) grp = (1 << (term - (1 + 3 * ((term - 2) / 3)))) - 1;
        // 1. grids of the columns and digits of T_{term-1}
        if (__any_sync(0xffffffffu, s_max[par][lane % NC] >= NOT_FINITE<T>)) {  // (the same in every warp)
            mark_not_finite<T>(a, par, s_max[par]);
            if (tid == 0) s_marked = 1;
            __syncthreads();
        }
        int ec;  // of column lane % NC
        const bool bad = opbad | __any_sync(0xffffffffu, !grid_exp<T>(s_max[par][lane % NC], D::EX_MIN, D::EX_MAX, ec));
        if (tid < NC) {
            s_e[tid] = ec;
            if (!F64) s_cf[tid] = bad ? 2.f : pow2(ec - 1, 0.f);
        }
        if (tid == 0) s_slow = bad;
        if (grp && tid < 3 * MAX_F) {
            const int i = tid / MAX_F, f = tid % MAX_F;  // term - 2 + i
            const double c = f < a.nf ? coef[(int64_t)f * a.coef_stride + term - 2 + i] : 0.0;
            s_c[i][f] = c;
            ff_split(c, s_ch[i][f], s_cl[i][f]);
        }
        if (!bad) {
            for (int b = cb0 + tid; b < cb1; b += NTH) {
                const int q = col_of(b), s = a.slot[b];
                T v[16];
                if constexpr (F64) {
#pragma unroll
                    for (int i = 0; i < 16; i += 2) {
                        const double2 u = __ldcg(reinterpret_cast<const double2 *>(R + (int64_t)b * BB + i));
                        v[i] = u.x;
                        v[i + 1] = u.y;
                    }
                } else {
#pragma unroll
                    for (int i = 0; i < 16; i += 4) {
                        const float4 u = __ldcg(reinterpret_cast<const float4 *>(R + (int64_t)b * BB + i));
                        v[i] = u.x;
                        v[i + 1] = u.y;
                        v[i + 2] = u.z;
                        v[i + 3] = u.w;
                    }
                }
                if (*(volatile int *)&s_marked) {
#pragma unroll
                    for (int i = 0; i < 16; ++i)
                        if (mag_bits(v[i]) >= NOT_FINITE<T>) v[i] = T(0);
                }
                uint4 *xs = X + s * XV;
                const int sw = 2 * (s & 3);
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    int e;
                    grid_exp<T>(s_max[par][4 * q + c], D::EX_MIN, D::EX_MAX, e);
                    const int col = (4 * q + c) & 7, tile = (4 * q + c) >> 3;
                    if constexpr (F64) {
                        uint32_t w0[6], w1[6];
                        panel_digits(w0, v[c], v[4 + c], e);
                        panel_digits(w1, v[8 + c], v[12 + c], e);
#pragma unroll
                        for (int i = 0; i < 3; ++i)
                            xs[8 * i + (col ^ sw)] = make_uint4(w0[2 * i], w1[2 * i], w0[2 * i + 1], w1[2 * i + 1]);
                    } else {
                        uint32_t w0[2], w1[2], b0, b1;
                        panel_digits(w0, b0, grid_value(v[c], e), grid_value(v[4 + c], e));
                        panel_digits(w1, b1, grid_value(v[8 + c], e), grid_value(v[12 + c], e));
                        xs[8 * tile + (col ^ sw)] = make_uint4(w0[0], w1[0], w0[1], w1[1]);
                        X2[s * 4 * XV + ((4 * q + c) ^ (8 * ((s >> 1) & 1)))] = b0 | (b1 << 16);
                    }
                }
            }
        }
        __syncthreads();
        if (tid < NC) s_max[par][tid] = 0u;  // next written by the step after the next
        if (tid == 0) s_marked = 0;

        // 2. the warp's groups
        uint32_t mx[NT][2];
        float gh = 0.f, gl = 0.f;  // <T, G>: FP32 as a double-float pair
        double gd = 0.0;
#pragma unroll
        for (int j = 0; j < NT; ++j) mx[j][0] = mx[j][1] = 0u;
        const int c0w = __ldg(a.wchunk + pid * (COL_NW + 1) + warp);
        const int r0w = __ldg(a.wrow + pid * (COL_NW + 1) + warp) - rbase, r1w = __ldg(a.wrow + pid * (COL_NW + 1) + warp + 1) - rbase;
        if (r0w < r1w) {
            // operator digits of a quad, rows g (half 0) and g + 8 (half 1)
            struct Op {
                uint32_t w[2][F64 ? 8 : 4];
            };
            const uint4 *ob = a.opd + (g & 3) * (F64 ? 2 : 1);
            auto load_h = [&](Op &o, uint2 w) {
                ld_row(o.w[0], ob, w.x >> COL_SLOT_BITS);
                ld_row(o.w[1], ob, w.y >> COL_SLOT_BITS);
            };
            // Two quads are on their way: quads go in pairs (even / odd) through two
            // register sets, each refilled two quads ahead as soon as its digits are
            // taken, its words four ahead (the lists end in padding).
            const uint2 *ep = reinterpret_cast<const uint2 *>(a.ent) + (int64_t)c0w * 8 + ((g >> 2) * 4 + t);
            uint2 wc[2] = {__ldg(ep), __ldg(ep + 8)}, wn[2] = {__ldg(ep + 16), __ldg(ep + 24)};
            Op h[2];
            load_h(h[0], wc[0]);
            load_h(h[1], wc[1]);
            ep += 32;
            int qi = 0;
            for (int r = r0w; r < r1w; ++r) {
                const uint2 rw = srow[r];
                const bool slow = *(volatile int *)&s_slow != 0;
                const int cnt = (int)(rw.y >> COL_SLOT_BITS);
                // sums of the group: rows g, g + 8 x columns 2t, 2t + 1 of each tile
                float dl[NT][2][4];      // digit sums kept in the accumulators (FP32: D_1, D_2; FP64: D_4, D_5)
                float fs[NT][4];         // FP32: the exact leading sums added up
                int is[4][4];            // FP64: the four exact digit sums
#pragma unroll
                for (int j = 0; j < NT; ++j)
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        fs[j][i] = 0.f;
#pragma unroll
                        for (int s = 0; s < 2; ++s) dl[j][s][i] = 0.f;
                    }
#pragma unroll
                for (int s = 0; s < 4; ++s)
#pragma unroll
                    for (int i = 0; i < 4; ++i) is[s][i] = 0;
                if (!slow) {
#pragma unroll 1
                    for (int k = 0; k < cnt; k += 2) {
                        float z[NT][F64 ? 4 : 1][4];  // exact sums of the pair
#pragma unroll
                        for (int o = 0; o < 2; ++o) {
                            const int sl = (int)(wc[o].x & SM);
                            const uint4 *xs = X + sl * XV + (g ^ (2 * (sl & 3)));
                            wc[o] = wn[o];
                            wn[o] = __ldg(ep + o * 8);
                            const float zero[4] = {0.f, 0.f, 0.f, 0.f};
                            if constexpr (!F64) {
                                uint32_t A0[4], A1[4], A2[4];
#pragma unroll
                                for (int i = 0; i < 4; ++i) {  // (half i % 2, pair i / 2)
                                    const uint32_t u = h[o].w[i & 1][i & 2], v = h[o].w[i & 1][(i & 2) + 1];
                                    A0[i] = f16_digits(u & 0x03ff03ffu);
                                    A1[i] = f16_digits(v & 0x03ff03ffu);
                                    A2[i] = spread_digit(u, v);
                                }
                                load_h(h[o], wc[o]);
                                const uint32_t *x2 = X2 + sl * 4 * XV;
                                const int g2 = g ^ (8 * ((sl >> 1) & 1));
                                uint32_t B[NT][3][2];
#pragma unroll
                                for (int j = 0; j < NT; ++j) {
                                    const uint4 xw = xs[8 * j];
                                    const uint32_t xb = x2[g2 ^ (8 * j)];
                                    B[j][0][0] = xw.x;
                                    B[j][0][1] = xw.y;
                                    B[j][1][0] = xw.z;
                                    B[j][1][1] = xw.w;
                                    B[j][2][0] = third_digits<0x4140>(xb);
                                    B[j][2][1] = third_digits<0x4342>(xb);
                                }
                                // (the leading sums of two quads, below 2^24, are exact)
#pragma unroll
                                for (int j = 0; j < NT; ++j) {
                                    if (o == 0) mma16816(z[j][0], A0, B[j][0], zero);
                                    else mma16816(z[j][0], A0, B[j][0], z[j][0]);
                                }
#pragma unroll
                                for (int j = 0; j < NT; ++j) mma16816(dl[j][0], A0, B[j][1], dl[j][0]);
#pragma unroll
                                for (int j = 0; j < NT; ++j) mma16816(dl[j][1], A0, B[j][2], dl[j][1]);
#pragma unroll
                                for (int j = 0; j < NT; ++j) mma16816(dl[j][0], A1, B[j][0], dl[j][0]);
#pragma unroll
                                for (int j = 0; j < NT; ++j) mma16816(dl[j][1], A1, B[j][1], dl[j][1]);
#pragma unroll
                                for (int j = 0; j < NT; ++j) mma16816(dl[j][1], A2, B[j][0], dl[j][1]);
                                if (o == 1) {
#pragma unroll
                                    for (int j = 0; j < NT; ++j)
#pragma unroll
                                        for (int i = 0; i < 4; ++i) fs[j][i] += z[j][0][i];
                                }
                            } else {
                                const uint4 x0 = xs[0], x1 = xs[8], x2 = xs[16];
                                const uint32_t B[6][2] = {{x0.x, x0.y}, {x0.z, x0.w}, {x1.x, x1.y},
                                                          {x1.z, x1.w}, {x2.x, x2.y}, {x2.z, x2.w}};
#pragma unroll
                                for (int i = 0; i < 6; ++i) {
                                    uint32_t A[4];
#pragma unroll
                                    for (int k2 = 0; k2 < 4; ++k2) {  // (half k2 % 2, pair k2 / 2)
                                        const uint32_t *hw = h[o].w[k2 & 1] + 2 * (k2 & 2);
                                        const uint32_t pw[4] = {hw[0], hw[1], hw[F64 ? 2 : 0], hw[F64 ? 3 : 0]};
                                        A[k2] = packed_digit(pw, i);
                                    }
                                    if (i >= 1) {  // D_6 into D_5's accumulator: the panel digit times 2^-10
                                        const uint32_t Bs[2] = {h2_fma(B[6 - i][0], 0x14001400u, 0u), h2_fma(B[6 - i][1], 0x14001400u, 0u)};
                                        mma16816(dl[0][1], A, Bs, dl[0][1]);
                                    }
#pragma unroll
                                    for (int s = i; s < 6; ++s) {
                                        if (s >= 4) mma16816(dl[0][s & 1], A, B[s - i], dl[0][s & 1]);
                                        else if (i == 0 && (o == 0 || s >= 2)) mma16816(z[0][F64 ? s : 0], A, B[s], zero);
                                        else mma16816(z[0][F64 ? s : 0], A, B[s - i], z[0][F64 ? s : 0]);
                                    }
                                    // (the sums of s = 0, 1 stay exact over two quads)
                                    if (i < 4 && (o == 1 || i >= 2)) {
#pragma unroll
                                        for (int e = 0; e < 4; ++e) is[i][e] += __float2int_rn(z[0][F64 ? i : 0][e]);
                                    }
                                }
                                load_h(h[o], wc[o]);
                            }
                        }
                        ep += 16;
                    }
                    // the digit sums as one value, in fs (FP32) or as the two halves
                    // of a double in is[0], is[1]
#pragma unroll
                    for (int j = 0; j < NT; ++j)
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            if constexpr (F64) {
                                const int64_t q = (((int64_t)is[0][i] * 1024 + is[1][i]) * 1024 + is[2][i]) * 1024 + is[3][i];
                                const double v = (double)q + (double)fmaf(dl[0][1][i], 0x1p-20f, dl[0][0][i] * 0x1p-10f);
                                is[0][i] = __double2hiint(v);
                                is[1][i] = __double2loint(v);
                            } else {
                                fs[j][i] = fmaf(fmaf(dl[j][1][i], 0x1p-10f, dl[j][0][i]), 0x1p-10f, fs[j][i]);
                            }
                        }
                } else {
                    // plain products (a call, so that they take no registers from the above)
                    T val[4 * NT];
                    plain_group<T>(a, opos, R, reinterpret_cast<const uint32_t *>(a.ent) + ((int64_t)c0w + qi) * COL_CW, cnt, lane, val);
                    qi += cnt;
#pragma unroll
                    for (int j = 0; j < NT; ++j)
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            if constexpr (F64) {
                                is[0][i] = __double2hiint(val[i]);
                                is[1][i] = __double2loint(val[i]);
                            } else {
                                fs[j][i] = val[4 * j + i];
                            }
                        }
                }
                // 3. the lane's elements: rows of atoms g/4 and g/4 + 2, scalar row
                // g % 4, block column 2 j + t/2, scalar columns 2 (t % 2) and + 1
                const int sl2[2] = {(int)((g >> 2) == 0 ? rw.x & SM : (rw.x >> COL_SLOT_BITS) & SM),
                                    (int)((g >> 2) == 0 ? (rw.x >> (2 * COL_SLOT_BITS)) & SM : rw.y & SM)};
                const int eo = 4 * (g & 3) + 2 * (t & 1);
                using GV = typename std::conditional<F64, double2, float4>::type;
#pragma unroll
                for (int hh = 0; hh < 2; ++hh) {
                    if (sl2[hh] == (int)SM) continue;
                    const int er = rexp[4 * sl2[hh] + (g & 3)];
                    const float rf = F64 || slow ? 1.f : pow2(er - 17, 0.f);  // (two exact factors)
                    // T_{term-2}, G and, in group steps, T_{term-1}, of the half's positions
                    int pos[NT];
                    V2 tm[NT], tk[NT], y[NT];
                    GV gv[NT];
#pragma unroll
                    for (int j = 0; j < NT; ++j) {
                        pos[j] = opos[sl2[hh] * P + 2 * j + (t >> 1)];
                        tm[j] = tk[j] = V2{};
                        gv[j] = GV{};
                        if (pos[j] < 0) continue;
                        const int64_t off = (int64_t)pos[j] * BB + eo;
                        tm[j] = __ldcg(reinterpret_cast<const V2 *>(C + off));
                        if (a.G) {
                            if constexpr (F64) gv[j] = __ldg(reinterpret_cast<const GV *>(a.G + (int64_t)a.tperm[pos[j]] * BB + eo));
                            else gv[j] = __ldcg(reinterpret_cast<const GV *>(a.Gp + off * 2));
                        }
                        if (grp) tk[j] = __ldcg(reinterpret_cast<const V2 *>(R + off));
                    }
#pragma unroll
                    for (int j = 0; j < NT; ++j) {
                        T w[2];
#pragma unroll
                        for (int cc = 0; cc < 2; ++cc) {
                            const int i = 2 * hh + cc;
                            T v, sc;
                            if constexpr (F64) {
                                v = __hiloint2double(is[0][i], is[1][i]);
                                sc = pow2(slow ? 1 : er + s_e[8 * j + 2 * t + cc] - 47, 0.0);
                            } else {
                                v = fs[j][i] * rf;
                                sc = s_cf[8 * j + 2 * t + cc];
                            }
                            w[cc] = mac(v, sc, cc ? -tm[j].y : -tm[j].x);
                            if constexpr (!F64) {
                                if (a.round_bf16) w[cc] = bf16r(w[cc]);
                            }
                        }
                        y[j].x = w[0];
                        y[j].y = w[1];
                        if (pos[j] < 0) continue;
                        *reinterpret_cast<V2 *>(C + (int64_t)pos[j] * BB + eo) = y[j];
                        mx[j][0] = max(mx[j][0], mag_bits(w[0]));
                        mx[j][1] = max(mx[j][1], mag_bits(w[1]));
                        if constexpr (F64) {
                            gd += gv[j].x * w[0] + gv[j].y * w[1];
                            if (grp) {
                                // the group's terms in order: T_{term-2}, T_{term-1}, T_term
                                const T tv[3][2] = {{tm[j].x, tm[j].y}, {tk[j].x, tk[j].y}, {w[0], w[1]}};
                                const int64_t at = (int64_t)a.tperm[pos[j]] * BB + eo;
                                for (int f = 0; f < a.nf; ++f) {
                                    double2 v = *reinterpret_cast<double2 *>(a.acc[f] + at);
#pragma unroll
                                    for (int i = 0; i < 3; ++i)
                                        if ((grp >> (2 - i)) & 1) {
                                            v.x += s_c[i][f] * tv[i][0];
                                            v.y += s_c[i][f] * tv[i][1];
                                        }
                                    *reinterpret_cast<double2 *>(a.acc[f] + at) = v;
                                }
                            }
                        } else if (a.G) {
                            ff_add_prod(gh, gl, w[0], gv[j].x, gv[j].y);
                            ff_add_prod(gh, gl, w[1], gv[j].z, gv[j].w);
                        }
                    }
                    if constexpr (!F64) {
                        // the same (the functions outside, so that the positions' loads go out
                        // together: four functions at 12,000 rows, 85.0 -> 82.9 ms)
                        for (int f = 0; grp && f < a.nf; ++f) {
                            float4 v[NT];
#pragma unroll
                            for (int j = 0; j < NT; ++j) {
                                if (pos[j] < 0) continue;
                                v[j] = __ldcg(reinterpret_cast<const float4 *>(a.accp[f] + ((int64_t)pos[j] * BB + eo) * 2));
                            }
#pragma unroll
                            for (int j = 0; j < NT; ++j) {
                                if (pos[j] < 0) continue;
                                const float tv[3][2] = {{tm[j].x, tm[j].y}, {tk[j].x, tk[j].y}, {y[j].x, y[j].y}};
#pragma unroll
                                for (int i = 0; i < 3; ++i)
                                    if ((grp >> (2 - i)) & 1) {
                                        ff_add_prod(v[j].x, v[j].y, tv[i][0], s_ch[i][f], s_cl[i][f]);
                                        ff_add_prod(v[j].z, v[j].w, tv[i][1], s_ch[i][f], s_cl[i][f]);
                                    }
                                *reinterpret_cast<float4 *>(a.accp[f] + ((int64_t)pos[j] * BB + eo) * 2) = v[j];
                            }
                        }
                    }
                }
            }
        }
        // the columns' largest elements, for the next step's grids
#pragma unroll
        for (int j = 0; j < NT; ++j)
#pragma unroll
            for (int cc = 0; cc < 2; ++cc) {
                uint32_t m = mx[j][cc];
#pragma unroll
                for (int o = 4; o < 32; o <<= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
                if (g == 0) atomicMax(&s_max[par ^ 1][8 * j + 2 * t + cc], m);
            }
        // 4. the panel's moments of this term: the warps' parts of <T, G>, and the
        // trace from the diagonal blocks
        if (a.want_mom) {
            const double w = warp_sum(F64 ? gd : (double)gh + (double)gl);
            if (lane == 0) red[warp] = w;
        }
        __syncthreads();
        if (a.want_mom && warp == 0) {
            double tr = 0.0;
            if (lane < 4 * nc) {
                const int q = lane >> 2, p = opos[s_dslot[q] * P + q];
                tr = (double)__ldcg(C + (int64_t)p * BB + 5 * (lane & 3));
            }
            tr = warp_sum(tr);
            const double gs = warp_sum(lane < COL_NW ? red[lane] : 0.0);
            if (lane == 0) {
                part[(int64_t)(term - a.tbase) * 2] = tr;
                part[(int64_t)(term - a.tbase) * 2 + 1] = gs;
            }
        }
    }
    // the FP32 accumulators back to the caller: FP64, BCSR order
    if constexpr (!F64) {
        if (a.t1 >= n) {
            for (int64_t e = (int64_t)cb0 * BB + tid; e < (int64_t)cb1 * BB; e += NTH) {
                const int64_t o = (int64_t)a.tperm[e / BB] * BB + e % BB;
                for (int f = 0; f < a.nf; ++f) {
                    const float2 v = __ldcg(reinterpret_cast<const float2 *>(a.accp[f]) + e);
                    a.acc[f][o] = (double)v.x + (double)v.y;
                }
            }
        }
    }
}

// mom[sys * stride + k] = sum over the system's panels of the partials of
// terms tbase .. tbase + nt - 1, in a fixed order: one thread block per term and
// system.
__global__ void __launch_bounds__(128) k_colmom(const double *part, int pstride, int tbase, int nt, const int32_t *sys_panel,
                                                const int32_t *n_terms, int n_single, int64_t mom_stride, double *mom,
                                                double *gmom) {
    __shared__ double sh[4];
    const int k = blockIdx.x, sy = blockIdx.y, n = n_terms ? n_terms[sy] : n_single;
    if (tbase + k >= n) return;
    double t = 0.0, g = 0.0;
    for (int p = sys_panel[sy] + threadIdx.x; p < sys_panel[sy + 1]; p += 128) {
        const double2 v = *reinterpret_cast<const double2 *>(part + ((int64_t)p * pstride + k) * 2);
        t += v.x;
        g += v.y;
    }
    t = block_sum<128>(t, sh);
    g = block_sum<128>(g, sh);
    if (threadIdx.x == 0) {
        if (mom) mom[sy * mom_stride + tbase + k] = t;
        if (gmom) gmom[sy * mom_stride + tbase + k] = g;
    }
}

// Steps per launch: a multiple of 3 (the accumulation groups), enough that the
// per-launch set-up of a panel (positions, zero digits) and the last wave of
// panels cost little, few enough that the moment table stays small.
constexpr int COL_STEPS = 96;

bool col_usable(const cheb_plan *plan, const cheb_bsr *Mt) {
    return plan->col.bound && plan->op_rp == Mt->row_ptr && plan->op_ci == Mt->col_idx && plan->col.nnzL == Mt->nnzb;
}

bool col_takes(const cheb_plan *plan, const cheb_bsr *Mt, const ColExpand &x, size_t ws_bytes) {
    if (!col_usable(plan, Mt) || ws_bytes < col_expand_ws(plan, Mt->nnzb)) return false;
    if (!wide_elements(plan->precision)) return true;
    // FP64 reads and writes the caller's accumulators and G in pairs
    uintptr_t at = x.gmoments ? reinterpret_cast<uintptr_t>(x.G) : 0;
    for (int f = 0; f < x.nf; ++f) at |= reinterpret_cast<uintptr_t>(x.acc[f]);
    return at % 16 == 0;
}

size_t col_expand_ws(const cheb_plan *plan, int64_t nnzL) {
    const bool wide = wide_elements(plan->precision);
    const size_t esz = wide ? 8 : 4;
    size_t b = 2 * align_up(plan->nnzb * BB * esz);
    b += align_up((size_t)(nnzL + 1) * (wide ? 128 : 64));
    if (!wide) b += (MAX_F + 1) * align_up(plan->nnzb * BB * 8);  // accumulators and G as float pairs
    b += align_up(plan->nbr * 16) + align_up(64);
    b += align_up((size_t)plan->col.n_panels * (COL_STEPS + 2) * 2 * sizeof(double));
    return b + 256;
}

template <typename T>
static int col_expand_t(const cheb_plan *plan, const cheb_bsr *Mt, const ColExpand &x, void *ws, size_t ws_bytes,
                        cudaStream_t s) {
    Carve cv = carve_aligned(ws, ws_bytes);
    const ColLists &c = plan->col;
    ColArgs a{};
    for (int i = 0; i < 2; ++i) a.T[i] = cv.take<T>(plan->nnzb * BB);
    uint4 *opd = cv.take<uint4>((Mt->nnzb + 1) * (sizeof(T) == 8 ? 8 : 4));
    if (sizeof(T) == 4) {
        for (int f = 0; f < MAX_F; ++f) a.accp[f] = cv.take<float>(plan->nnzb * BB * 2);
        a.Gp = cv.take<float>(plan->nnzb * BB * 2);
    }
    int32_t *opexp = cv.take<int32_t>(4 * plan->nbr), *opflag = cv.take<int32_t>(16);
    a.part = cv.take<double>((size_t)c.n_panels * (COL_STEPS + 2) * 2);
    if (!cv.fits()) return fail(CHEB_ERR_NOSPACE, "cheb_expand: workspace %zu too small", ws_bytes);
    CHEB_CUDA(cudaMemsetAsync(opflag, 0, 64, s));
    k_opdig<T><<<(unsigned)((plan->nbr + 1 + 7) / 8), 256, 0, s>>>(Mt->row_ptr, (const double *)Mt->vals, plan->nbr,
                                                                  Mt->nnzb, x.round_bf16, Dig<T>::OP_MIN, Dig<T>::OP_MAX,
                                                                  opd, opexp, opflag);
    CHEB_TRY(check_launch("k_opdig"));
    a.panels = c.d_panels;
    a.order = c.d_order;
    a.wchunk = c.d_wchunk;
    a.wrow = c.d_wrow;
    a.rows = c.d_rows;
    a.ent = c.d_ent;
    a.slot = c.d_slot;
    a.rp = plan->rp;
    a.ci = plan->ci;
    a.tperm = plan->d_tperm;
    a.Lrp = Mt->row_ptr;
    a.Lci = Mt->col_idx;
    a.Lv = (const double *)Mt->vals;
    a.nnzL = Mt->nnzb;
    a.opd = opd;
    a.opexp = opexp;
    a.opflag = opflag;
    a.n_terms = x.n_terms;
    a.n_single = x.max_terms;
    a.nf = x.nf;
    for (int f = 0; f < x.nf; ++f) a.acc[f] = x.acc[f];
    a.coef = x.coef;
    a.coef_off = x.coef_off;
    a.coef_stride = x.coef_stride;
    a.G = x.gmoments ? x.G : nullptr;
    a.pstride = COL_STEPS + 2;
    a.want_mom = x.moments || a.G;
    a.round_bf16 = x.round_bf16;
    const size_t smem = col_layout(c.P).total(c.max_union);
    auto fn = k_colstep<T>;
    CHEB_TRY(allow_shared(fn));
    for (int t0 = 2; t0 == 2 || t0 < x.max_terms; t0 += COL_STEPS) {
        a.t0 = t0;
        a.t1 = std::min(t0 + COL_STEPS, x.max_terms);
        a.tbase = t0 == 2 ? 0 : t0;
        fn<<<(unsigned)c.n_panels, COL_NW * 32, smem, s>>>(a);
        CHEB_TRY(check_launch("k_colstep"));
        if (a.want_mom) {
            const int nt = a.t1 - a.tbase;
            k_colmom<<<dim3(nt, plan->nsys), 128, 0, s>>>(a.part, a.pstride, a.tbase, nt, c.d_sys_panel, x.n_terms,
                                                          x.max_terms, x.mom_stride, x.moments, a.G ? x.gmoments : nullptr);
            CHEB_TRY(check_launch("k_colmom"));
        }
    }
    return CHEB_OK;
}

int col_expand(const cheb_plan *plan, const cheb_bsr *Mt, const ColExpand &x, void *ws, size_t ws_bytes, cudaStream_t s) {
    if (ws_bytes < col_expand_ws(plan, Mt->nnzb))
        return fail(CHEB_ERR_NOSPACE, "cheb_expand: workspace %zu < %zu", ws_bytes, col_expand_ws(plan, Mt->nnzb));
    return wide_elements(plan->precision) ? col_expand_t<double>(plan, Mt, x, ws, ws_bytes, s)
                                          : col_expand_t<float>(plan, Mt, x, ws, ws_bytes, s);
}

// ---------------------------------------------------------------------------
// Host: the column kernel's panels and work streams for operator pattern
// (lrp, lci).  Per panel: the union of its columns' rows (slot = rank), in groups
// of four: the first row left, then three times the row among the next COL_WINDOW
// left that brings the fewest new slots for its length; per group the slots K with
// an operator block in any of its rows, ascending (neighbouring slots are often
// neighbouring blocks of the operator), eight to two quads (col_places), and per
// slot of a quad the operator block of each row, or the zero block; groups dealt to the NW warps by decreasing quad count, each to the warp with the
// fewest quads so far; per warp its groups' quads in one stream and its group list.

struct ColCounts {
    std::vector<int64_t> chunks, rows;
    std::vector<int32_t> max_row;
};

static void col_fill(const ColLists &c, const std::vector<int64_t> &rp, const std::vector<int32_t> &ci,
                     const std::vector<int64_t> &lrp, const std::vector<int32_t> &lci, int64_t nbr, int64_t p0,
                     int64_t p1, bool count_only, ColCounts &cnt, const std::vector<int64_t> &chunk_off,
                     const std::vector<int64_t> &row_off, std::vector<int32_t> &wchunk, std::vector<int32_t> &wrow,
                     std::vector<uint32_t> &rows, std::vector<uint32_t> &ent, std::vector<uint16_t> &slot) {
    const int NW = c.NW;
    const uint32_t zero_blk = (uint32_t)lci.size();  // the appended zero block
    std::vector<int32_t> stamp(nbr, -1), slot_of(nbr, -1), uni, order;
    std::vector<int> work, left;
    std::vector<std::array<int, 4>> groups;
    std::vector<uint32_t> bits;  // [union row][words] operator slots
    std::vector<int64_t> load(NW);
    std::vector<std::vector<int32_t>> wgroups(NW);
    for (int64_t p = p0; p < p1; ++p) {
        const int32_t j0 = c.h_panels[4 * p], nc = c.h_panels[4 * p + 1];
        uni.clear();
        for (int32_t q = 0; q < nc; ++q)
            for (int64_t e = rp[j0 + q]; e < rp[j0 + q + 1]; ++e)
                if (stamp[ci[e]] != (int32_t)p) {
                    stamp[ci[e]] = (int32_t)p;
                    uni.push_back(ci[e]);
                }
        std::sort(uni.begin(), uni.end());
        const int nu = (int)uni.size(), ng = (nu + 3) / 4, nw = (nu + 31) / 32;
        for (int u = 0; u < nu; ++u) slot_of[uni[u]] = u;
        bits.assign((size_t)nu * nw, 0u);
        for (int u = 0; u < nu; ++u)
            for (int64_t e = lrp[uni[u]]; e < lrp[uni[u] + 1]; ++e)
                if (stamp[lci[e]] == (int32_t)p) {
                    const int s = slot_of[lci[e]];
                    bits[(size_t)u * nw + (s >> 5)] |= 1u << (s & 31);
                }
        left.resize(nu);
        std::iota(left.begin(), left.end(), 0);
        groups.assign(ng, {-1, -1, -1, -1});
        work.assign(ng, 2);
        int32_t mr = 0;
        int64_t total = 0;
        std::vector<std::vector<uint32_t>> merged(ng);
        for (int i = 0; i < ng; ++i) {
            std::vector<uint32_t> &cur = merged[i];
            cur.assign(nw, 0u);
            for (int a = 0; a < 4 && !left.empty(); ++a) {
                int best = 0, bc = INT32_MAX;
                for (int k = 0; a > 0 && k < std::min<int>(COL_WINDOW, (int)left.size()); ++k) {
                    int cost = 0;
                    for (int w = 0; w < nw; ++w) {
                        const uint32_t b = bits[(size_t)left[k] * nw + w];
                        cost += 2 * __builtin_popcount(b & ~cur[w]) - __builtin_popcount(b);
                    }
                    if (cost < bc) {
                        bc = cost;
                        best = k;
                    }
                }
                const int u = left[best];
                left.erase(left.begin() + best);
                groups[i][a] = u;
                for (int w = 0; w < nw; ++w) cur[w] |= bits[(size_t)u * nw + w];
            }
            int n = 0;
            for (int w = 0; w < nw; ++w) n += __builtin_popcount(cur[w]);
            work[i] = std::max(2, (n + 7) / 8 * 2);
            mr = std::max(mr, work[i]);
            total += work[i];
        }
        if (count_only) {
            cnt.chunks[p] = total;
            cnt.rows[p] = ng;
            cnt.max_row[p] = mr;
            continue;
        }
        order.resize(ng);
        std::iota(order.begin(), order.end(), 0);
        std::stable_sort(order.begin(), order.end(), [&](int32_t x, int32_t y) { return work[x] > work[y]; });
        std::fill(load.begin(), load.end(), 0);
        for (auto &v : wgroups) v.clear();
        for (const int32_t i : order) {
            const int w = (int)(std::min_element(load.begin(), load.end()) - load.begin());
            load[w] += work[i];
            wgroups[w].push_back(i);
        }
        for (int32_t q = 0; q < nc; ++q)
            for (int64_t e = rp[j0 + q]; e < rp[j0 + q + 1]; ++e) slot[e] = (uint16_t)slot_of[ci[e]];
        int64_t ch = chunk_off[p], ro = row_off[p];
        for (int w = 0; w < NW; ++w) {
            wchunk[p * (NW + 1) + w] = (int32_t)ch;
            wrow[p * (NW + 1) + w] = (int32_t)ro;
            std::sort(wgroups[w].begin(), wgroups[w].end());
            for (const int32_t i : wgroups[w]) {
                const int quads = work[i];
                uint32_t sl[4];
                for (int a = 0; a < 4; ++a) sl[a] = groups[i][a] >= 0 ? (uint32_t)groups[i][a] : (1u << COL_SLOT_BITS) - 1u;
                rows[2 * ro] = sl[0] | (sl[1] << COL_SLOT_BITS) | (sl[2] << (2 * COL_SLOT_BITS));
                rows[2 * ro + 1] = sl[3] | ((uint32_t)quads << COL_SLOT_BITS);
                ++ro;
                uint32_t *out = ent.data() + ch * COL_CW;
                auto word = [&](int pl, int a) -> uint32_t & {
                    return out[(pl >> 2) * COL_CW + ((a & 1) * 4 + (pl & 3)) * 2 + (a >> 1)];
                };
                const std::vector<uint32_t> &cur = merged[i];
                std::vector<int> place(32 * nw, -1);
                std::vector<uint16_t> list;
                for (int s = 0; s < nu; ++s)
                    if ((cur[s >> 5] >> (s & 31)) & 1u) list.push_back((uint16_t)s);
                for (int c8 = 0; c8 < quads / 2; ++c8) {
                    uint8_t at[8];
                    unsigned taken = 0u;
                    const int n = std::max(0, std::min<int>(8, (int)list.size() - 8 * c8));
                    col_places(list.data() + 8 * c8, n, at);
                    for (int k = 0; k < n; ++k) {
                        const int s = list[8 * c8 + k];
                        place[s] = 8 * c8 + at[k];
                        taken |= 1u << at[k];
                        for (int a = 0; a < 4; ++a) word(place[s], a) = (zero_blk << COL_SLOT_BITS) | (uint32_t)s;
                    }
                    for (int k = 0; k < 8; ++k)
                        if (!((taken >> k) & 1u))
                            for (int a = 0; a < 4; ++a)
                                word(8 * c8 + k, a) = (zero_blk << COL_SLOT_BITS) | (uint32_t)((k & 3) < nu ? k & 3 : 0);
                }
                for (int a = 0; a < 4 && groups[i][a] >= 0; ++a)
                    for (int64_t e = lrp[uni[groups[i][a]]]; e < lrp[uni[groups[i][a]] + 1]; ++e)
                        if (stamp[lci[e]] == (int32_t)p) {
                            const int s = slot_of[lci[e]];
                            word(place[s], a) = ((uint32_t)e << COL_SLOT_BITS) | (uint32_t)s;
                        }
                ch += quads;
            }
        }
        wchunk[p * (NW + 1) + NW] = (int32_t)ch;
        wrow[p * (NW + 1) + NW] = (int32_t)ro;
    }
}

// Union rows a panel of the column kernel may hold: shared memory, and
// col_max_union.
int32_t col_ucap(int P) {
    const ColLayout lay = col_layout(P);
    return std::min((CHEB_MAX_DYN_SMEM - 1024 - lay.off_x) / lay.slot_bytes, col_max_union(P));
}

// Whether the column kernel's lists are built for an operator of nnzL blocks
// (see COL_ROW_MIN) whose index fits an entry word.
bool col_wanted(const cheb_plan *plan, int64_t nnzL) {
    if (nnzL + 1 >= ((int64_t)1 << (32 - COL_SLOT_BITS))) return false;
    return !wide_elements(plan->precision) || nnzL >= COL_ROW_MIN * plan->nbr;
}

int col_build(cheb_plan *plan, const std::vector<int64_t> &rp, const std::vector<int32_t> &ci,
              const std::vector<int64_t> &lrp, const std::vector<int32_t> &lci) {
    ColLists c;
    const bool wide = wide_elements(plan->precision);
    c.P = col_width(plan->precision);
    c.NW = COL_NW;
    c.nnzL = (int64_t)lci.size();
    const int64_t nbr = plan->nbr, nnzb = plan->nnzb;
    c.ucap = col_ucap(c.P);
    if (!col_wanted(plan, c.nnzL)) return CHEB_ERR_NOSPACE;
    // panels: greedy along the columns of each system while the union fits
    std::vector<int32_t> stamp(nbr, -1);
    c.h_sys_panel.clear();
    for (int sy = 0; sy < plan->nsys; ++sy) {
        int64_t j = plan->h_sys_col[sy], panel = c.n_panels;
        c.h_sys_panel.push_back((int32_t)panel);
        while (j < plan->h_sys_col[sy + 1]) {
            int32_t cnt = 0, ncols = 0;
            const int64_t j0 = j;
            while (j < plan->h_sys_col[sy + 1] && ncols < c.P) {
                int32_t add = 0;
                for (int64_t p = rp[j]; p < rp[j + 1]; ++p) add += stamp[ci[p]] != (int32_t)panel;
                if (cnt + add > c.ucap) break;
                for (int64_t p = rp[j]; p < rp[j + 1]; ++p) stamp[ci[p]] = (int32_t)panel;
                cnt += add;
                ++ncols;
                ++j;
            }
            if (ncols == 0) return CHEB_ERR_NOSPACE;  // a single column does not fit: no column kernel
            c.h_panels.insert(c.h_panels.end(), {(int32_t)j0, ncols, cnt, sy});
            c.max_union = std::max(c.max_union, cnt);
            ++panel;
        }
        c.n_panels = panel;
    }
    c.h_sys_panel.push_back((int32_t)c.n_panels);
    const int64_t np = c.n_panels;
    ColCounts cnt;
    cnt.chunks.assign(np, 0);
    cnt.rows.assign(np, 0);
    cnt.max_row.assign(np, 0);
    std::vector<int64_t> chunk_off(np + 1, 0), row_off(np + 1, 0);
    std::vector<int32_t> wchunk(np * (c.NW + 1)), wrow(np * (c.NW + 1));
    std::vector<uint32_t> rows, ent;
    std::vector<uint16_t> slot(nnzb);
    const int nth = (int)std::max<int64_t>(1, std::min<int64_t>({(int64_t)std::thread::hardware_concurrency(), 16, np}));
    auto run = [&](bool count_only) {
        std::vector<std::thread> th;
        for (int t = 0; t < nth; ++t) {
            const int64_t p0 = np * t / nth, p1 = np * (t + 1) / nth;
            th.emplace_back([&, p0, p1] {
                col_fill(c, rp, ci, lrp, lci, nbr, p0, p1, count_only, cnt, chunk_off, row_off, wchunk, wrow, rows, ent, slot);
            });
        }
        for (auto &x : th) x.join();
    };
    run(true);
    for (int64_t p = 0; p < np; ++p) {
        chunk_off[p + 1] = chunk_off[p] + cnt.chunks[p];
        row_off[p + 1] = row_off[p] + cnt.rows[p];
        c.max_row = std::max(c.max_row, cnt.max_row[p]);
    }
    if ((chunk_off[np] + COL_TAIL) * COL_CW >= (int64_t)INT32_MAX || (wide && c.max_row > COL_MAX_QUADS64)) return CHEB_ERR_NOSPACE;
    c.n_entries = (chunk_off[np] + COL_TAIL) * COL_CW;
    rows.resize(2 * row_off[np]);
    ent.resize(c.n_entries, 0u);
    run(false);
    c.h_wchunk.swap(wchunk);
    c.h_wrow.swap(wrow);
    c.h_rows.swap(rows);
    c.h_ent.swap(ent);
    c.h_slot.swap(slot);
    c.n_rows = (int64_t)c.h_rows.size();
    c.n_slot = (int64_t)c.h_slot.size();
    c.n_sys = (int64_t)c.h_sys_panel.size();
    c.h_order = col_order(cnt.chunks);
    c.built = true;
    plan->col = std::move(c);
    return CHEB_OK;
}

// Thread blocks start in the order of their index, one per SM at a time, so the panels
// that start last should be the short ones: the LAST panels with the fewest quads (two
// per SM) go last, longest first, the others in their own order, in which neighbours
// share operator rows in L2.  250 panels FP32: 10.1 -> 8.4 ms; 500 and 771 panels FP64:
// 24.5 -> 22.2 and 91.0 -> 88.5 ms.  Beyond eight panels per SM all stay in their own
// order: the last wave is a small part, and the short panels, far apart, miss L2 more
// (2,502 panels FP32: 128.8 -> 131.7 ms).
std::vector<int32_t> col_order(const std::vector<int64_t> &quads) {
    constexpr size_t SMS = 152, LAST = 2 * SMS;
    const size_t np = quads.size();
    std::vector<int32_t> by(np), order;
    std::iota(by.begin(), by.end(), 0);
    if (np > 8 * SMS) return by;
    std::stable_sort(by.begin(), by.end(), [&](int32_t x, int32_t y) { return quads[x] > quads[y]; });
    const size_t first = np - std::min(np, LAST);
    order.assign(by.begin(), by.begin() + first);
    std::sort(order.begin(), order.end());
    order.insert(order.end(), by.begin() + first, by.end());
    return order;
}

int col_bind(ColLists &c, Carve &cv, cudaStream_t s) {
    if (!c.built) return CHEB_OK;
    if (c.device) {
        // lists built on the device: one copy of their block into the workspace
        // (the same carve order, so every array keeps its offset)
        char *dst = cv.take<char>(c.bytes());
        if (!cv.fits()) return fail(CHEB_ERR_NOSPACE, "cheb_plan_bind_operator: workspace too small");
        CHEB_CUDA(cudaMemcpyAsync(dst, c.tmp, c.bytes(), cudaMemcpyDeviceToDevice, s));
        const ptrdiff_t d = dst - static_cast<char *>(c.tmp);
        c.d_panels = reinterpret_cast<int32_t *>(reinterpret_cast<char *>(c.d_panels) + d);
        c.d_wchunk = reinterpret_cast<int32_t *>(reinterpret_cast<char *>(c.d_wchunk) + d);
        c.d_wrow = reinterpret_cast<int32_t *>(reinterpret_cast<char *>(c.d_wrow) + d);
        c.d_rows = reinterpret_cast<uint32_t *>(reinterpret_cast<char *>(c.d_rows) + d);
        c.d_ent = reinterpret_cast<uint32_t *>(reinterpret_cast<char *>(c.d_ent) + d);
        c.d_slot = reinterpret_cast<uint16_t *>(reinterpret_cast<char *>(c.d_slot) + d);
        c.d_sys_panel = reinterpret_cast<int32_t *>(reinterpret_cast<char *>(c.d_sys_panel) + d);
        c.d_order = reinterpret_cast<int32_t *>(reinterpret_cast<char *>(c.d_order) + d);
        return CHEB_OK;
    }
    c.d_panels = cv.take<int32_t>(c.h_panels.size());
    c.d_wchunk = cv.take<int32_t>(c.h_wchunk.size());
    c.d_wrow = cv.take<int32_t>(c.h_wrow.size());
    c.d_rows = cv.take<uint32_t>(std::max<size_t>(c.h_rows.size(), 1));
    c.d_ent = cv.take<uint32_t>(std::max<size_t>(c.h_ent.size(), 1));
    c.d_slot = cv.take<uint16_t>(c.h_slot.size());
    c.d_sys_panel = cv.take<int32_t>(c.h_sys_panel.size());
    c.d_order = cv.take<int32_t>(c.h_order.size());
    if (!cv.fits()) return fail(CHEB_ERR_NOSPACE, "cheb_plan_bind_operator: workspace too small");
    CHEB_CUDA(cudaMemcpyAsync(c.d_panels, c.h_panels.data(), c.h_panels.size() * 4, cudaMemcpyHostToDevice, s));
    CHEB_CUDA(cudaMemcpyAsync(c.d_wchunk, c.h_wchunk.data(), c.h_wchunk.size() * 4, cudaMemcpyHostToDevice, s));
    CHEB_CUDA(cudaMemcpyAsync(c.d_wrow, c.h_wrow.data(), c.h_wrow.size() * 4, cudaMemcpyHostToDevice, s));
    if (!c.h_rows.empty())
        CHEB_CUDA(cudaMemcpyAsync(c.d_rows, c.h_rows.data(), c.h_rows.size() * 4, cudaMemcpyHostToDevice, s));
    if (!c.h_ent.empty())
        CHEB_CUDA(cudaMemcpyAsync(c.d_ent, c.h_ent.data(), c.h_ent.size() * 4, cudaMemcpyHostToDevice, s));
    CHEB_CUDA(cudaMemcpyAsync(c.d_slot, c.h_slot.data(), c.h_slot.size() * 2, cudaMemcpyHostToDevice, s));
    CHEB_CUDA(cudaMemcpyAsync(c.d_sys_panel, c.h_sys_panel.data(), c.h_sys_panel.size() * 4, cudaMemcpyHostToDevice, s));
    CHEB_CUDA(cudaMemcpyAsync(c.d_order, c.h_order.data(), c.h_order.size() * 4, cudaMemcpyHostToDevice, s));
    return CHEB_OK;
}

void col_free(ColLists &c) {
    if (c.tmp) cudaFree(c.tmp);
    c.tmp = nullptr;
}

void col_release_host(ColLists &c) {
    col_free(c);  // (after the stream has been synchronised)
    std::vector<int32_t>().swap(c.h_wchunk);
    std::vector<int32_t>().swap(c.h_wrow);
    std::vector<uint32_t>().swap(c.h_rows);
    std::vector<uint32_t>().swap(c.h_ent);
    std::vector<uint16_t>().swap(c.h_slot);
    c.bound = c.built;
}

}  // namespace cheb
