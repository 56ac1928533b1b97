// Masked products C = alpha P(A B) + beta D of FP64 plans with long rows (Eq. 3's
// product by itself: orthogonalisation, post-processing and Newton-Schulz steps), on
// the tensor cores by the digits of colstep.cu.
//
// What bounds it.  On the FP64 pipe (k_step) a 4x4 block product is 64 multiply-adds at
// two per cycle and SM.  As digits it is 26 mma for 16 rows, 16 inner and 8 columns.
// The left operand is often a matrix on the output pattern (an inverse root, a density
// matrix), for which no quad lists are kept (the operator's are a few hundred MB
// already at 6,000 rows), so a warp finds its quads itself: a table of its four rows
// over the panel's union rows, from which it takes the fours of neighbouring union
// rows that any of its rows has a block in.  That is a tenth of the work; neighbouring
// union rows are often neighbours in space, so the fours are 60 % full.
// Measured (GB300), orthogonalisation and post-processing at 1,500 atoms, 10 / 14 bohr
// (one product with the operator on the left, three on the output pattern): 66.5 ms
// on the FP64 pipe, 14.5 ms here.  Error against 64 bits 4.2e-16 -> 4.0e-16.  Values beyond
// the grids or not finite, one product at 1,000 atoms: 6.3 ms there, 7.0 ms here.
//
// One thread block per panel of two columns (one after the other where their union
// does not fit): the union of their rows, the columns of B as packed digits in shared
// memory, 32 bytes per union row and scalar column; a warp takes groups of four
// neighbouring union rows.  The left operand's digits are formed once per call in the
// plan's workspace; calls on streams that share a place there wait for each other.
#include <mutex>

#include "common.cuh"
#include "digits.cuh"
#include "kernels.cuh"
#include "plan.cuh"

namespace cheb {

constexpr int PR_NW = 16;
// Grid exponents that the products take, of either operand.
constexpr int PR_EX = 400;
// Quads whose exact digit sums (at most 2^24 a quad) stay below 2^31.
constexpr int PR_CHUNK = 126;

struct ProdArgs {
    const int64_t *rp;
    const int32_t *ci, *tperm, *panels;
    const int64_t *Lrp;
    const int32_t *Lci;
    const double *Lv;
    int64_t nnzL;
    const uint4 *opd;
    const int32_t *opexp, *opflag;
    const double *R, *D;
    double *C;
    double alpha, beta;
    int32_t cap;  // union rows that fit (a multiple of 4)
    int32_t nw;   // words of the union's bitmap
};

struct ProdLayout {
    int off_pos, off_x, off_tab, off_q, off_bits;
};
__host__ __device__ constexpr ProdLayout prod_layout(int cap) {
    ProdLayout L{};
    int o = cap * 4;  // union list
    L.off_pos = o;    // block position of (union row, column)
    o += cap * 8;
    o = (o + 127) / 128 * 128;
    L.off_x = o;  // packed digits: chunk (rows 0 1, rows 2 3) and column of each union row
    o += (cap + 4) * 256;
    L.off_tab = o;  // per warp: offset of the block (row of the group, union row) in its operator row
    o += PR_NW * 4 * (cap + 4) * 2;
    L.off_q = o;  // per warp: quads with a block
    o += PR_NW * (cap / 4 + 4);
    L.off_bits = (o + 15) / 16 * 16;  // the union as a bitmap, 8 bytes a word of 32 block rows
    return L;
}
// Union rows that fit beside the bitmap (0: none).
static int prod_cap(const cheb_plan *plan) {
    const int64_t room = CHEB_MAX_DYN_SMEM - 1024 - (plan->nbr + 31) / 32 * 8;
    int cap = (plan->max_union + 3) & ~3;
    while (cap > 0 && prod_layout(cap).off_bits > room) cap -= 4;
    return cap;
}

// The digits resolve a column when, for one of its rows, the sum of |products| is at
// least 2^-PR_RESOLVE of the row's and the column's grids multiplied: the grids' error is
// then at most K u of that sum, like that of FP64 sums.  Where none is -- the large
// elements of the rows meet the small ones of the column, so that the scales cancel --
// the panel is done once more in plain FP64.  A result of that size shows it for free; a
// panel with a column of smaller ones gets its sums of |leading digits| formed (one mma
// instead of 26; sums that cancel, as in the product of a density matrix with a column
// that it nearly annihilates, are no reason to take FP64: 0.5 ms a panel at 800 rows).
constexpr int PR_RESOLVE = 6;

// The products of one group in plain FP64 (an element beyond the digits' grids, or a
// column that they do not resolve).
__device__ __noinline__ void prod_plain(const ProdArgs &a, const int32_t *opos, const uint16_t *tab, int ts, int nu,
                                        const int64_t *base, int lane, double *out) {
    const int g = lane >> 2, t = lane & 3;
    for (int i = 0; i < 4; ++i) out[i] = 0.0;
    for (int s = 0; s < nu; ++s) {
        const uint32_t id[2] = {tab[(g >> 2) * ts + s], tab[((g >> 2) + 2) * ts + s]};
        const int p = opos[2 * s + (t >> 1)];
        if ((id[0] & id[1]) == 0xffffu || p < 0) continue;
        double2 x[4];
#pragma unroll
        for (int m = 0; m < 4; ++m) x[m] = __ldg(reinterpret_cast<const double2 *>(a.R + (int64_t)p * BB + 4 * m + 2 * (t & 1)));
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            if (id[h] == 0xffffu) continue;
            const double *hv = a.Lv + (base[h] + id[h]) * BB + 4 * (g & 3);
#pragma unroll
            for (int m = 0; m < 4; ++m) {
                const double w = __ldg(hv + m);
                out[2 * h] = fma(w, x[m].x, out[2 * h]);
                out[2 * h + 1] = fma(w, x[m].y, out[2 * h + 1]);
            }
        }
    }
}

// The sums of |leading digits| of one group, where the mma has them (in units of 2^-18 of
// the grids multiplied).
__device__ __noinline__ void prod_scale(const uint4 *ob, const uint4 *X, const uint16_t *tl, int ts, const unsigned char *ql,
                                        int cnt, uint32_t base0, uint32_t base1, uint32_t none, int g, int t, float *out) {
    float z[4] = {0.f, 0.f, 0.f, 0.f};
    for (int k = 0; k < cnt; ++k) {
        const int q = ql[k];
        const uint32_t i0 = tl[4 * q], i1 = tl[2 * ts + 4 * q];
        uint32_t w[2][8];
        ld_row(w[0], ob, i0 == 0xffffu ? none : base0 + i0);
        ld_row(w[1], ob, i1 == 0xffffu ? none : base1 + i1);
        const uint4 *xs = X + (4 * q + t) * 16 + (g ^ (2 * t));
        constexpr uint32_t D0 = 0x03ff03ffu, ABS = 0x7fff7fffu;
        const uint32_t A[4] = {f16_digits(w[0][0] & D0) & ABS, f16_digits(w[1][0] & D0) & ABS,
                               f16_digits(w[0][4] & D0) & ABS, f16_digits(w[1][4] & D0) & ABS};
        const uint32_t B[2] = {f16_digits(xs[0].x & D0) & ABS, f16_digits(xs[8].x & D0) & ABS};
        mma16816(z, A, B, z);
    }
    for (int i = 0; i < 4; ++i) out[i] = z[i];
}

__global__ void __launch_bounds__(PR_NW * 32, 1) k_product(const __grid_constant__ ProdArgs a) {
    constexpr int NTH = PR_NW * 32;
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ uint32_t s_max[8];
    __shared__ int s_e[8];
    __shared__ int s_slow, s_big[8], wsum[32];  // s_big: columns that the digits resolve
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, cap = a.cap, ts = cap + 4;
    const ProdLayout lay = prod_layout(cap);
    int32_t *ulist = reinterpret_cast<int32_t *>(smem), *opos = reinterpret_cast<int32_t *>(smem + lay.off_pos);
    uint4 *X = reinterpret_cast<uint4 *>(smem + lay.off_x);
    uint2 *bits = reinterpret_cast<uint2 *>(smem + lay.off_bits);
    uint16_t *tab = reinterpret_cast<uint16_t *>(smem + lay.off_tab) + warp * 4 * ts;
    unsigned char *ql = smem + lay.off_q + warp * (cap / 4 + 4);
    const unsigned lt = (1u << lane) - 1u;
    const int j0 = a.panels[2 * blockIdx.x], nj = a.panels[2 * blockIdx.x + 1];
    for (int q0 = 0, nc = 0; q0 < nj; q0 += nc) {
        // 1. the union of the columns' rows as a bitmap with ranks, the second column only
        // if it still fits
        nc = min(2, nj - q0);
        const int64_t r0 = a.rp[j0 + q0], r1 = a.rp[j0 + q0 + 1], r2 = a.rp[j0 + q0 + nc];
        int nu = 0;
        int64_t re = r2;  // end of the blocks taken
        while (true) {
            __syncthreads();  // (the pass before is done with shared memory)
            for (int w = tid; w < a.nw; w += NTH) bits[w] = make_uint2(0u, 0u);
            __syncthreads();
            for (int64_t b = r0 + tid; b < re; b += NTH) atomicOr(&bits[a.ci[b] >> 5].x, 1u << (a.ci[b] & 31));
            __syncthreads();
            const int per = (a.nw + NTH - 1) / NTH, w0 = min(a.nw, tid * per), w1 = min(a.nw, w0 + per);
            int n = 0;
            for (int w = w0; w < w1; ++w) n += __popc(bits[w].x);
            int run = block_excl_scan<PR_NW>(n, wsum, &nu);
            for (int w = w0; w < w1; ++w) {
                bits[w].y = (unsigned)run;
                run += __popc(bits[w].x);
            }
            if (nu <= a.cap) break;  // (every thread finds the same; a single column fits)
            nc = 1;
            re = r1;
        }
        const int nu4 = (nu + 3) & ~3;
        // 2. positions and the columns' largest elements, then their digits
        for (int i = tid; i < (nu4 + 4) * 16; i += NTH) X[i] = make_uint4(0x82008200u, 0x02000200u, 0x82008200u, 0x02000200u);
        for (int i = tid; i < 2 * nu; i += NTH) opos[i] = -1;
        if (tid < 8) s_max[tid] = 0u;
        if (tid == 0) s_slow = *a.opflag != 0;
        __syncthreads();
        for (int64_t b = r0 + tid; b < re; b += NTH) {
            const int q = b >= r1, K = a.ci[b], s = rank_of(bits, K);
            const int p = a.tperm[b];
            ulist[s] = K;
            opos[2 * s + q] = p;
            uint32_t m[4] = {0u, 0u, 0u, 0u};
#pragma unroll
            for (int e = 0; e < 16; e += 2) {
                const double2 v = *reinterpret_cast<const double2 *>(a.R + (int64_t)p * BB + e);
                m[e & 3] = max(m[e & 3], mag_bits(v.x));
                m[(e & 3) + 1] = max(m[(e & 3) + 1], mag_bits(v.y));
            }
#pragma unroll
            for (int c = 0; c < 4; ++c) atomicMax(&s_max[4 * q + c], m[c]);
        }
        __syncthreads();
        if (tid < 8) {
            int e;
            if (!grid_exp<double>(s_max[tid], -PR_EX, PR_EX, e)) s_slow = 1;
            s_e[tid] = e;
            s_big[tid] = 0;
        }
        __syncthreads();
        enum { DIGITS, SCALE, PLAIN };
        int mode = s_slow != 0 ? PLAIN : DIGITS;
        if (mode == DIGITS) {
            for (int i = tid; i < 2 * nu; i += NTH) {
                const int p = opos[i], s = i >> 1, q = i & 1, sw = 2 * (s & 3);
                if (p < 0) continue;
                double v[16];
#pragma unroll
                for (int e = 0; e < 16; e += 2) {
                    const double2 u = *reinterpret_cast<const double2 *>(a.R + (int64_t)p * BB + e);
                    v[e] = u.x;
                    v[e + 1] = u.y;
                }
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    const int col = 4 * q + c, e = s_e[col];
                    uint32_t w[4];
                    pack_pair(w, v[c], v[4 + c], e);
                    X[s * 16 + (col ^ sw)] = make_uint4(w[0], w[1], w[2], w[3]);
                    pack_pair(w, v[8 + c], v[12 + c], e);
                    X[s * 16 + 8 + (col ^ sw)] = make_uint4(w[0], w[1], w[2], w[3]);
                }
            }
        }
        __syncthreads();
        // 3. the warp's groups of four union rows
        const int g = lane >> 2, t = lane & 3;
        const uint4 *ob = a.opd + (g & 3) * 2;
        while (true) {
            for (int gi = warp; 4 * gi < nu; gi += PR_NW) {
                __syncwarp();
                for (int i = lane; i < ts; i += 32) reinterpret_cast<uint64_t *>(tab)[i] = ~0ull;
                __syncwarp();
                for (int r = 0; r < 4 && 4 * gi + r < nu; ++r) {
                    const int64_t b = a.Lrp[ulist[4 * gi + r]];
                    const int len = (int)(a.Lrp[ulist[4 * gi + r] + 1] - b);
                    for (int i = lane; i < len; i += 32) {
                        const int s = rank_of(bits, __ldg(a.Lci + b + i));
                        if (s >= 0) tab[r * ts + s] = (uint16_t)i;
                    }
                }
                __syncwarp();
                int64_t base[2];
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int u = 4 * gi + (g >> 2) + 2 * h;
                    base[h] = u < nu ? a.Lrp[ulist[u]] : 0;
                }
                double val[4] = {0.0, 0.0, 0.0, 0.0};
                if (mode == PLAIN) {
                    prod_plain(a, opos, tab, ts, nu, base, lane, val);
                } else {
                    int cnt = 0;
                    for (int b = 0; b < nu4 / 4; b += 32) {
                        const int q = b + lane;
                        bool any = false;
                        if (q < nu4 / 4) {
                            uint64_t all = ~0ull;
#pragma unroll
                            for (int r = 0; r < 4; ++r) all &= *reinterpret_cast<const uint64_t *>(tab + r * ts + 4 * q);
                            any = all != ~0ull;
                        }
                        const unsigned m = __ballot_sync(0xffffffffu, any);
                        if (any) ql[cnt + __popc(m & lt)] = (unsigned char)q;
                        cnt += __popc(m);
                    }
                    // quads go in pairs: an empty one (beyond the union) fills up the last
                    if (lane == 0) ql[cnt] = (unsigned char)(nu4 / 4);
                    cnt = (cnt + 1) & ~1;
                    __syncwarp();
                    struct Op {
                        uint32_t w[2][8];
                    };
                    const uint32_t base0 = (uint32_t)base[0], base1 = (uint32_t)base[1], none = (uint32_t)a.nnzL;
                    const uint16_t *tl = tab + (g >> 2) * ts + t;
                    auto load_h = [&](Op &o, int k) {
                        const int q = ql[min(k, cnt - 1)];
                        const uint32_t i0 = tl[4 * q], i1 = tl[2 * ts + 4 * q];
                        ld_row(o.w[0], ob, i0 == 0xffffu ? none : base0 + i0);
                        ld_row(o.w[1], ob, i1 == 0xffffu ? none : base1 + i1);
                    };
                    if (mode == SCALE) {
                        float z[4];
                        prod_scale(ob, X, tl, ts, ql, cnt, base0, base1, none, g, t, z);
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            const int u = 4 * gi + (g >> 2) + 2 * (i >> 1);
                            if (u < nu && opos[2 * u + (t >> 1)] >= 0 && z[i] >= (float)(1 << (18 - PR_RESOLVE)))
                                s_big[2 * t + (i & 1)] = 1;
                        }
                        continue;
                    }
                    Op h[2];
                    if (cnt > 0) {
                        load_h(h[0], 0);
                        load_h(h[1], 1);
                    }
                    for (int k0 = 0; k0 < cnt; k0 += PR_CHUNK) {
                        const int k1 = min(cnt, k0 + PR_CHUNK);
                        float dl[2][4];
                        int is[4][4];
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            dl[0][i] = dl[1][i] = 0.f;
#pragma unroll
                            for (int s = 0; s < 4; ++s) is[s][i] = 0;
                        }
#pragma unroll 1
                        for (int k = k0; k < k1; k += 2) {
                            float z[4][4];
#pragma unroll
                            for (int o = 0; o < 2; ++o) {
                                const uint4 *xs = X + (4 * ql[k + o] + t) * 16 + (g ^ (2 * t));
                                const uint4 x0 = xs[0], x1 = xs[8];
                                const uint32_t w0[4] = {x0.x, x0.y, x0.z, x0.w}, w1[4] = {x1.x, x1.y, x1.z, x1.w};
                                uint32_t B[6][2];
#pragma unroll
                                for (int i = 0; i < 6; ++i) {
                                    B[i][0] = packed_digit(w0, i);
                                    B[i][1] = packed_digit(w1, i);
                                }
                                const float zero[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
                                for (int i = 0; i < 6; ++i) {
                                    uint32_t A[4];
#pragma unroll
                                    for (int e = 0; e < 4; ++e) {  // (half e % 2, pair e / 2)
                                        const uint32_t *hw = h[o].w[e & 1] + 2 * (e & 2);
                                        const uint32_t pw[4] = {hw[0], hw[1], hw[2], hw[3]};
                                        A[e] = packed_digit(pw, i);
                                    }
#pragma unroll
                                    for (int s = i; s < 6; ++s) {
                                        if (s >= 4) mma16816(dl[s & 1], A, B[s - i], dl[s & 1]);
                                        else if (i == 0 && (o == 0 || s >= 2)) mma16816(z[s], A, B[s], zero);
                                        else mma16816(z[s], A, B[s - i], z[s]);
                                    }
                                    // (the sums of s = 0, 1 stay exact over two quads)
                                    if (i >= 1) {  // D_6 into D_5's accumulator: the panel digit times 2^-10
                                        const uint32_t Bs[2] = {h2_fma(B[6 - i][0], 0x14001400u, 0u), h2_fma(B[6 - i][1], 0x14001400u, 0u)};
                                        mma16816(dl[1], A, Bs, dl[1]);
                                    }
                                    if (i < 4 && (o == 1 || i >= 2)) {
#pragma unroll
                                        for (int e = 0; e < 4; ++e) is[i][e] += __float2int_rn(z[i][e]);
                                    }
                                }
                                load_h(h[o], k + o + 2);
                            }
                        }
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            const int64_t q = (((int64_t)is[0][i] * 1024 + is[1][i]) * 1024 + is[2][i]) * 1024 + is[3][i];
                            val[i] += (double)q + (double)fmaf(dl[1][i], 0x1p-20f, dl[0][i] * 0x1p-10f);
                        }
                    }
                }
                // 4. the lane's elements (as in colstep.cu)
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int u = 4 * gi + (g >> 2) + 2 * h;
                    if (u >= nu) continue;
                    const int p = opos[2 * u + (t >> 1)];
                    if (p < 0) continue;
                    double y[2];
#pragma unroll
                    for (int c = 0; c < 2; ++c) {
                        y[c] = val[2 * h + c];
                        if (mode == PLAIN) continue;
                        if (fabs(y[c]) >= (double)(1ll << (48 - PR_RESOLVE))) s_big[2 * t + c] = 1;
                        y[c] *= pow2(a.opexp[4 * ulist[u] + (g & 3)] + s_e[2 * t + c] - 48, 0.0);
                    }
                    const int64_t at = (int64_t)p * BB + 4 * (g & 3) + 2 * (t & 1);
                    double2 v = make_double2(a.alpha * y[0], a.alpha * y[1]);
                    if (a.D) {
                        const double2 d = *reinterpret_cast<const double2 *>(a.D + at);
                        v = make_double2(fma(a.alpha, y[0], a.beta * d.x), fma(a.alpha, y[1], a.beta * d.y));
                    }
                    *reinterpret_cast<double2 *>(a.C + at) = v;
                }
            }
            if (mode == PLAIN) break;
            __syncthreads();
            bool done = true;
            for (int c = 0; c < 8; ++c) done &= s_max[c] == 0u || s_big[c] != 0;
            if (done) break;
            ++mode;  // (every thread finds the same; a lane writes over its own results)
            __syncthreads();
        }
    }
}

// The digits of one left operand, and how many of them a plan keeps: streams with their
// own run side by side, which pays while a product leaves SMs idle (50 panels, eight
// streams: 0.24 against 0.64 ms with one), so within 24 MB
// (150 atoms; 300 atoms are 150 panels, and eight streams gain 6 %).
static size_t prod_slot_bytes(const cheb_plan *plan, int64_t nnzL) {
    const int64_t n = std::max(nnzL, plan->nnzb);
    return align_up((size_t)(n + 1) * 128) + align_up(plan->nbr * 16) + align_up(64);
}
static int prod_slots(const cheb_plan *plan, int64_t nnzL) {
    return (int)std::clamp<size_t>(((size_t)24 << 20) / prod_slot_bytes(plan, nnzL), 1, PROD_SLOTS);
}
size_t prod_bytes(const cheb_plan *plan, int64_t nnzL) {
    if (plan->precision != CHEB_F64 || !plan->col.built || plan->nbr > 65535 || plan->max_row > prod_cap(plan)) return 0;
    return prod_slots(plan, nnzL) * prod_slot_bytes(plan, nnzL) + align_up(plan->n_panels * 8);
}

// The panels go to the device in the order of their launch: by the square of their
// union, as the column kernel's by their quads.
int prod_bind(cheb_plan *plan, Carve &cv, std::vector<int32_t> &panels, cudaStream_t s) {
    const size_t bytes = prod_bytes(plan, plan->col.nnzL);
    plan->prod_ws = bytes ? cv.take<char>(bytes) : nullptr;
    if (!cv.fits()) return fail(CHEB_ERR_NOSPACE, "cheb_plan_bind_operator: workspace too small");
    if (!bytes) return CHEB_OK;
    std::vector<int64_t> work;
    for (const int32_t u : plan->h_union) work.push_back((int64_t)u * u);
    for (const int32_t p : col_order(work)) panels.insert(panels.end(), {plan->h_panels[2 * p], plan->h_panels[2 * p + 1]});
    char *at = static_cast<char *>(plan->prod_ws) + bytes - align_up(plan->n_panels * 8);
    CHEB_CUDA(cudaMemcpyAsync(at, panels.data(), panels.size() * 4, cudaMemcpyHostToDevice, s));
    return CHEB_OK;
}

// Long rows (those of the column kernel's lists: the FP64 pipe bounds them, and the
// kernels for short rows keep their bits) of the operator or of a matrix on the output
// pattern, in arrays aligned for the loads; not while the stream is captured, since a
// graph's replays cannot be ordered with other calls' use of the digits.
bool prod_takes(const cheb_plan *plan, const cheb_bsr *L, const double *R, const double *D, const double *C,
                cudaStream_t s) {
    if (!plan->prod_ws || !plan->op_bound) return false;
    const bool op = L->row_ptr == plan->op_rp && L->col_idx == plan->op_ci && L->nnzb == plan->col.nnzL;
    const bool out = L->row_ptr == plan->rp && L->col_idx == plan->ci && L->nnzb == plan->nnzb;
    if (!op && !out) return false;
    const uintptr_t at = reinterpret_cast<uintptr_t>(R) | reinterpret_cast<uintptr_t>(D) | reinterpret_cast<uintptr_t>(C);
    if (at % 16) return false;
    cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(s, &st) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return st == cudaStreamCaptureStatusNone;
}

int prod_run(const cheb_plan *plan, const cheb_bsr *L, const double *R, double alpha, const double *D, double beta,
             double *C, cudaStream_t s) {
    const int64_t n = std::max(plan->col.nnzL, plan->nnzb);
    const size_t slot_bytes = prod_slot_bytes(plan, plan->col.nnzL);
    const int slots = prod_slots(plan, plan->col.nnzL);
    CHEB_TRY(allow_shared(k_product));
    // the stream's digits, or the next ones in turn; one user of them at a time: this call
    // waits, on its stream, for their last
    std::lock_guard<std::mutex> lock(plan->prod_mx);
    int slot = 0;
    while (slot < slots && !(plan->prod_slot[slot].done && plan->prod_slot[slot].stream == s)) ++slot;
    if (slot == slots) {
        slot = plan->prod_next % slots;
        plan->prod_next = (slot + 1) % slots;
    }
    cheb_plan::ProdSlot &used = plan->prod_slot[slot];
    Carve cv(static_cast<char *>(plan->prod_ws) + slot * slot_bytes, slot_bytes);
    ProdArgs a{};
    uint4 *opd = cv.take<uint4>((n + 1) * 8);
    int32_t *opexp = cv.take<int32_t>(4 * plan->nbr), *flag = cv.take<int32_t>(16);
    a.panels = reinterpret_cast<const int32_t *>(static_cast<char *>(plan->prod_ws) + slots * slot_bytes);
    a.rp = plan->rp;
    a.ci = plan->ci;
    a.tperm = plan->d_tperm;
    a.Lrp = L->row_ptr;
    a.Lci = L->col_idx;
    a.Lv = static_cast<const double *>(L->vals);
    a.nnzL = L->nnzb;
    a.opd = opd;
    a.opexp = opexp;
    a.opflag = flag;
    a.R = R;
    a.D = D;
    a.C = C;
    a.alpha = alpha;
    a.beta = beta;
    a.cap = prod_cap(plan);
    a.nw = (int32_t)((plan->nbr + 31) / 32);
    const int smem = prod_layout(a.cap).off_bits + a.nw * 8;
    if (!used.done) CHEB_CUDA(cudaEventCreateWithFlags(&used.done, cudaEventDisableTiming));
    else CHEB_CUDA(cudaStreamWaitEvent(s, used.done, 0));
    used.stream = s;
    CHEB_CUDA(cudaMemsetAsync(flag, 0, 64, s));
    k_opdig<double><<<(unsigned)((plan->nbr + 1 + 7) / 8), 256, 0, s>>>(L->row_ptr, a.Lv, plan->nbr, L->nnzb, 0, -PR_EX, PR_EX, opd,
                                                                      opexp, flag);
    CHEB_TRY(check_launch("k_opdig"));
    k_product<<<(unsigned)plan->n_panels, PR_NW * 32, smem, s>>>(a);
    const int rc = check_launch("k_product");
    CHEB_CUDA(cudaEventRecord(used.done, s));
    return rc;
}

}  // namespace cheb
