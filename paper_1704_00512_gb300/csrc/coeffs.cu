// Chebyshev coefficients (Eq. 4), degree selection (Eq. 6), the penalty trace
// (Eq. 5) and the mu bisection on the trace functional (Sec. "Fermi Operator
// Expansion"), all in FP64.
#include <cooperative_groups.h>

#include <algorithm>
#include <mutex>
#include <vector>

#include "common.cuh"

namespace cheb {

constexpr int GRID_UNIFORM = 8193;

struct FuncArr {
    cheb_func f[8];
};

__device__ __forceinline__ double fermi(double x, double mu, double kT) {
    return 1.0 / (1.0 + exp((x - mu) / kT));
}

// f(x) for the unscaled variable x; sigma/tau map x into [-1,1] (Eq. 2).
__device__ double feval(const cheb_func &f, double x, double sigma, double tau) {
    switch (f.kind) {
        case CHEB_FERMI: return fermi(x, f.mu, f.kT);
        case CHEB_ERFC: return 0.5 * erfc((x - f.mu) / f.kT);
        case CHEB_POWER: return pow(x, f.a);
        case CHEB_INTERVAL: return fermi(x, f.hi, f.kT) - fermi(x, f.lo, f.kT);
        case CHEB_PENALTY: {
            const double xs = sigma * (x - tau), al = fabs(f.a);
            return exp(-al * (xs + 1.0)) - exp(al * (xs - 1.0));
        }
        default: return 0.0;
    }
}

// x_k = cos(pi (k+1/2)/n) / sigma + tau: the k-th Chebyshev node mapped back (Eq. 4).
__device__ __forceinline__ double node(int k, int n, double sigma, double tau) {
    return cos(M_PI * (k + 0.5) / n) / sigma + tau;
}

// cos(pi j (2k+1) / (2n)) with the angle reduced exactly modulo 4n.
__device__ __forceinline__ double dct_cos(int64_t j, int64_t k, int64_t n) {
    const int64_t idx = (j * (2 * k + 1)) % (4 * n);
    return cos(M_PI * (double)idx / (2.0 * (double)n));
}

// The candidates of one batch, passed by value: their term counts, the divisors of
// the two-step transform, and the first of their values in arrays that hold them one
// after the other (total values per function).
constexpr int CAND_MAX = 96;
struct Cand {
    int n[CAND_MAX], n1[CAND_MAX];
    int64_t off[CAND_MAX];
    int nc;
    int64_t total;
};

// Cosine tables cos(pi i / (2n)), i < 4n, of every candidate n (tab + 4 off[c]).
__global__ void k_cos_table(Cand d, double *tab) {
    const int c = blockIdx.y;
    const int64_t n = d.n[c];
    double *t = tab + 4 * d.off[c];
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < 4 * n; i += (int64_t)gridDim.x * blockDim.x)
        t[i] = cospi((double)i / (2.0 * (double)n));
}

// f at the nodes of every (function, candidate) pair, in the order of the
// transform below: the even nodes ascending, then the odd ones descending.
__global__ void k_nodes(FuncArr F, Cand d, double sigma, double tau, double *fv) {
    const int fc = blockIdx.y, f = fc / d.nc, c = fc % d.nc;
    const int n = d.n[c];
    double *v = fv + f * d.total + d.off[c];
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < n; k += gridDim.x * blockDim.x)
        v[k & 1 ? n - 1 - k / 2 : k / 2] = feval(F.f[f], node(k, n, sigma, tau), sigma, tau);
}

// The coefficients c_j = (2/n) sum_k f_k cos(pi j (k+1/2)/n) (Eq. 4) as the real part
// of a discrete Fourier transform (J. Makhoul, IEEE Trans. ASSP 28, 27 (1980)):
// with v = (f_0, f_2, ..., f_3, f_1), c_j = (2/n) Re(e^{-i pi j/2n} sum_k v_k
// e^{-2 pi i j k/n}), and that transform in two steps for n = n1 n2, k = n2 a + b,
// j = j1 + n1 j2 (J. Cooley and J. Tukey, Math. Comput. 19, 297 (1965)):
//     Y[j1][b] = e^{-2 pi i j1 b/n} sum_a v[n2 a + b] e^{-2 pi i a j1/n1},
//     V[j1 + n1 j2] = sum_b Y[j1][b] e^{-2 pi i b j2/n2},
// so n (n1 + n2) products instead of n^2, n1 the largest divisor of n up to its
// square root.  Every cosine and sine is an entry of the table of cos(pi i/2n).
// (The plain sum, a gather of the table per product, took 4 ms for one function
// at n = 9216, and 20 ms for all candidates of a degree search up to 16384; now
// 0.1 and 0.5 ms.  Against long doubles the coefficients' error went from 0.6e-15 to
// 0.4e-15 at n = 300 and from 3.6e-15 to 0.9e-15 at n = 9216.)
__device__ __forceinline__ double2 twiddle(const double *t, int64_t m, int64_t n) {  // e^{-2 pi i m/n}, 0 <= m < n
    return make_double2(t[4 * m], -t[4 * m >= n ? 4 * m - n : 4 * m + 3 * n]);
}
__global__ void k_dft1(const double *fv, Cand d, const double *tab, double2 *Y) {
    const int fc = blockIdx.y, f = fc / d.nc, c = fc % d.nc;
    const int n = d.n[c], n1 = d.n1[c], n2 = n / n1;
    const double *v = fv + f * d.total + d.off[c], *t = tab + 4 * d.off[c];
    double2 *y = Y + f * d.total + d.off[c];
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const int j1 = i / n2, b = i % n2;
        double re = 0.0, im = 0.0;
        int m = 0;  // a j1 mod n1
        for (int a = 0; a < n1; ++a) {
            const double2 w = twiddle(t, (int64_t)n2 * m, n);
            const double x = v[(int64_t)n2 * a + b];
            re = fma(x, w.x, re);
            im = fma(x, w.y, im);
            m += j1;
            if (m >= n1) m -= n1;
        }
        const double2 w = twiddle(t, (int64_t)j1 * b, n);  // j1 b < n1 n2
        y[i] = make_double2(re * w.x - im * w.y, re * w.y + im * w.x);
    }
}
constexpr int DFT_LANES = 8;
__global__ void k_dft2(const double2 *Y, Cand d, const double *tab, double *cv) {
    const int fc = blockIdx.y, f = fc / d.nc, c = fc % d.nc;
    const int n = d.n[c], n1 = d.n1[c], n2 = n / n1;
    const double *t = tab + 4 * d.off[c];
    const double2 *y = Y + f * d.total + d.off[c];
    double *out = cv + f * d.total + d.off[c];
    // A prime n is one long sum per j (n1 = 1): eight lanes share it, and since the values
    // are real, so that V[n - j] is the conjugate of V[j], half the sums do (n = 9973:
    // 3.30 -> 0.56 ms; 3.11 by the plain sum).
    const int lanes = n1 == 1 ? DFT_LANES : 1, count = n1 == 1 ? n / 2 + 1 : n;
    for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < (int64_t)count * lanes; k += (int64_t)gridDim.x * blockDim.x) {
        const int i = (int)(k / lanes), b0 = (int)(k % lanes);
        const int j1 = i / n2, j2 = i % n2, step = (int)((int64_t)lanes * j2 % n2);
        double re = 0.0, im = 0.0;
        int m = (int)((int64_t)b0 * j2 % n2);  // b j2 mod n2
        for (int b = b0; b < n2; b += lanes) {
            const double2 w = twiddle(t, (int64_t)n1 * m, n), u = y[(int64_t)j1 * n2 + b];
            re = fma(u.x, w.x, fma(-u.y, w.y, re));
            im = fma(u.x, w.y, fma(u.y, w.x, im));
            m += step;
            if (m >= n2) m -= n2;
        }
        if (n1 == 1) {
            const unsigned mine = 0xffu << (threadIdx.x & 24);
#pragma unroll
            for (int o = 1; o < DFT_LANES; o <<= 1) {
                re += __shfl_xor_sync(mine, re, o);
                im += __shfl_xor_sync(mine, im, o);
            }
            if (b0 != 0) continue;
        }
        const int j = j1 + n1 * j2;
        out[j] = (2.0 / n) * (re * t[j] + im * t[j + 3 * n]);  // e^{-i pi j/2n}
        if (n1 == 1 && j > 0) out[n - j] = (2.0 / n) * (re * t[n - j] - im * t[4 * n - j]);
    }
}

__device__ __forceinline__ unsigned long long dbits(double v) { return __double_as_longlong(v); }

struct Pairs {
    int n, at[8];
};
__device__ __forceinline__ void max_to(double emax, double fm, unsigned long long *e, unsigned long long *f) {
    // warp max then one atomic per warp; over non-negative doubles on their bit
    // patterns (order-independent)
    for (int o = 16; o > 0; o >>= 1) {
        emax = fmax(emax, __shfl_xor_sync(0xffffffffu, emax, o));
        fm = fmax(fm, __shfl_xor_sync(0xffffffffu, fm, o));
    }
    if ((threadIdx.x & 31) == 0) {
        if (e) atomicMax(e, dbits(emax));
        if (f) atomicMax(f, dbits(fm));
    }
}

// max |p_n(x) - f(x)| over the degree grid: 8193 uniform points on [-1,1] plus the
// 2n+1 extrema of T_{2n}, by the scalar recursion T_{j+1} = 2 x T_j - T_{j-1} with
// explicit roundings.  One (function, candidate) pair per blockIdx.y: pairs.at[y].
__global__ void k_fit_error(FuncArr F, const double *cv, Cand d, Pairs pairs, double sigma, double tau,
                            unsigned long long *errmax) {
    const int fc = pairs.at[blockIdx.y], f = fc / d.nc, c = fc % d.nc;
    const int n = d.n[c];
    const double *cc = cv + f * d.total + d.off[c];
    const int npts = GRID_UNIFORM + 2 * n + 1;
    double emax = 0.0;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < npts; i += gridDim.x * blockDim.x) {
        double x;
        if (i < GRID_UNIFORM) x = -1.0 + i * (2.0 / (GRID_UNIFORM - 1));
        else x = cos(M_PI * (double)(i - GRID_UNIFORM) / (2.0 * n));
        double Tm = 1.0, T = x;
        double p = __dmul_rn(0.5 * cc[0], Tm);
        if (n > 1) p = __dadd_rn(p, __dmul_rn(cc[1], T));
        const double x2 = __dmul_rn(2.0, x);
        for (int j = 2; j < n; ++j) {
            const double Tn = __dsub_rn(__dmul_rn(x2, T), Tm);
            Tm = T;
            T = Tn;
            p = __dadd_rn(p, __dmul_rn(cc[j], T));
        }
        const double fx = feval(F.f[f], x / sigma + tau, sigma, tau);
        emax = fmax(emax, fabs(p - fx));
    }
    max_to(emax, 0.0, errmax + fc, nullptr);
}
// The same but for rounding, with a fourth of the FP64 operations (two per lane and
// cycle bound it) and none of the serial chain: x goes with -x, whose sums are the even
// terms' plus or minus the odd ones'; a warp takes a point, lane l the terms l, l + 32,
// ... by T_{j+32} = 2 T_32 T_j - T_{j-32}; fused multiply-adds.  With stride > 1 only
// every stride-th uniform point.  Also the largest |f| met.  pairs.n = 0: the pair is
// blockIdx.y.  (By the plain recursion, a thread per point: 0.6 ms where this takes
// 0.2, at 6,000 terms, and 1.2 ms for the 513 points of eight candidates around 12,000.)
__global__ void __launch_bounds__(256) k_fit_estimate(FuncArr F, const double *cv, Cand d, Pairs pairs, int stride,
                                                      double sigma, double tau, unsigned long long *errmax,
                                                      unsigned long long *fabsmax) {
    const int fc = pairs.n ? pairs.at[blockIdx.y] : blockIdx.y, f = fc / d.nc, c = fc % d.nc;
    const int n = d.n[c], lane = threadIdx.x & 31;
    const double *cc = cv + f * d.total + d.off[c];
    constexpr int HALF = GRID_UNIFORM / 2;  // the point x = 0
    const int npts = stride > 1 ? HALF / stride + 1 : HALF + n + 2;
    double emax = 0.0, fm = 0.0;
    for (int k = blockIdx.x * 8 + (threadIdx.x >> 5); k < npts; k += gridDim.x * 8) {
        const int i = k * stride;
        const double x = i <= HALF ? -1.0 + i * (2.0 / (GRID_UNIFORM - 1)) : cos(M_PI * (double)(i - HALF - 1) / (2.0 * n));
        const double th = acos(x), t2 = 2.0 * cos(32.0 * th);
        double a = cos(lane * th), b = cos((lane + 32) * th), s = 0.0;
        for (int j = lane; j < n; j += 32) {
            s = fma(j == 0 ? 0.5 * cc[0] : __ldg(cc + j), a, s);
            const double t = fma(t2, b, -a);
            a = b;
            b = t;
        }
        const double odd = lane & 1 ? -s : s;  // the term's sign at -x
        const double pp = warp_sum(s), pn = warp_sum(odd);
        if (lane == 0) {
            const double fp = feval(F.f[f], x / sigma + tau, sigma, tau), fn = feval(F.f[f], -x / sigma + tau, sigma, tau);
            emax = fmax(emax, fmax(fabs(pp - fp), fabs(pn - fn)));
            fm = fmax(fm, fmax(fabs(fp), fabs(fn)));
        }
    }
    max_to(emax, fm, errmax + fc, fabsmax + fc);
}
// max |f(x)| over the same grid, without the polynomial.
__global__ void k_fit_scale(FuncArr F, Cand d, double sigma, double tau, unsigned long long *fabsmax) {
    const int fc = blockIdx.y, f = fc / d.nc, c = fc % d.nc;
    const int n = d.n[c], npts = GRID_UNIFORM + 2 * n + 1;
    double fm = 0.0;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < npts; i += gridDim.x * blockDim.x) {
        double x;
        if (i < GRID_UNIFORM) x = -1.0 + i * (2.0 / (GRID_UNIFORM - 1));
        else x = cos(M_PI * (double)(i - GRID_UNIFORM) / (2.0 * n));
        fm = fmax(fm, fabs(feval(F.f[f], x / sigma + tau, sigma, tau)));
    }
    max_to(0.0, fm, nullptr, fabsmax + fc);
}

// out[f][j], j < n_max: the coefficients of candidate ci (n terms), 0 beyond.
__global__ void k_pick(const double *cv, Cand d, int ci, int n, int n_max, double *out) {
    const int f = blockIdx.y;
    const double *c = cv + f * d.total + d.off[ci];
    for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < n_max; j += gridDim.x * blockDim.x)
        out[(int64_t)f * n_max + j] = j < n ? c[j] : 0.0;
}

// Penalty coefficients at n terms (Eq. 4 for Eq. 5), one thread per coefficient, the
// nodes in order.  f is formed once per node and, while they fit shared memory, the
// cosines cos(pi i/2n) once per table entry (the values that dct_cos has), by every
// thread block for its PEN_J coefficients.  (Two exponentials and a cosine for each of
// the n^2 products took 4 ms at n = 512; now 0.05 ms.)  The order of the sums stays what it is: the
// trace is a small difference of large terms, and its rounding with it.
constexpr int PEN_J = 32, PEN_NT = 256, PEN_TAB = 1024;
__global__ void __launch_bounds__(PEN_NT) k_penalty_coeffs(double alpha, int n, double *c) {
    __shared__ double tab[4 * PEN_TAB], fk[PEN_TAB];
    const cheb_func f{CHEB_PENALTY, 0, 0, alpha, 0, 0};
    const bool small = n <= PEN_TAB;
    if (small)
        for (int i = threadIdx.x; i < 4 * n; i += PEN_NT) tab[i] = cos(M_PI * (double)i / (2.0 * (double)n));
    const int j = blockIdx.x * PEN_J + threadIdx.x;
    const bool mine = threadIdx.x < PEN_J && j < n;
    double s = 0.0;
    for (int k0 = 0; k0 < n; k0 += PEN_TAB) {
        const int k1 = min(n, k0 + PEN_TAB);
        __syncthreads();
        // scaled variable directly: sigma = 1, tau = 0
        for (int k = k0 + threadIdx.x; k < k1; k += PEN_NT) fk[k - k0] = feval(f, node(k, n, 1.0, 0.0), 1.0, 0.0);
        __syncthreads();
        if (!mine) continue;
        if (small) {
            int idx = j;  // j (2k+1) mod 4n
            for (int k = 0; k < n; ++k) {
                s += fk[k] * tab[idx];
                idx += 2 * j;
                if (idx >= 4 * n) idx -= 4 * n;
            }
        } else {
            for (int k = k0; k < k1; ++k) s += fk[k - k0] * dct_cos(j, k, n);
        }
    }
    if (mine) c[j] = (2.0 / n) * s;
}

template <int NT>
__global__ void k_dot_terms(const double *c, const double *t, int n, double *out) {
    __shared__ double sh[NT / 32];
    double s = 0.0;
    for (int k = threadIdx.x; k < n; k += NT) s += (k == 0 ? 0.5 * c[0] : c[k]) * t[k];
    double r = block_sum<NT>(s, sh);
    if (threadIdx.x == 0) *out = r;
}

// w_i = (2/n) [g_0/2 + sum_{k>=1} g_k cos(pi k (i+1/2)/n)], so that
// N(mu) = sum_i f(x_i; mu) w_i equals c_0(mu) g_0/2 + sum_k c_k(mu) g_k
// (the two finite sums of Eq. 4 and Eq. 1 swapped).
//
// cos(k phi_i), phi_i = pi (i+1/2)/n, by angle addition: k = k0 + r, r < CW_R, with
// cos(r phi) and sin(r phi) of the thread's node in registers, so that a term takes
// two multiply-adds; the angle of k0 advances by rotation and is taken afresh (exact
// reduction) every CW_FRESH blocks.  Node n-1-i has the angle pi - phi_i: its sum
// is the even terms' minus the odd terms', so only half the nodes are computed.  A
// thread block takes 32 nodes and splits k over its warps.  (A cosine per term, with
// a 64-bit modulus, took 9 ms at n = 9216; now 0.33 ms.)
constexpr int CW_R = 8, CW_FRESH = 16, CW_NW = 16;
__global__ void __launch_bounds__(CW_NW * 32) k_count_weights(const double *g, int n, double *w) {
    __shared__ double se[CW_NW][33], so[CW_NW][33];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int half = (n + 1) / 2, i = min(blockIdx.x * 32 + lane, half - 1);
    const int64_t n4 = 4 * (int64_t)n, step = 2 * i + 1;
    double cr[CW_R], sr[CW_R];
#pragma unroll
    for (int r = 0; r < CW_R; ++r) sincospi((double)(r * step % n4) / (2.0 * n), &sr[r], &cr[r]);
    double rc, rs;  // the rotation by CW_R steps
    sincospi((double)(CW_R * step % n4) / (2.0 * n), &rs, &rc);
    const int nb = (n + CW_R - 1) / CW_R, per = (nb + CW_NW - 1) / CW_NW;
    double even = 0.0, odd = 0.0, kc = 1.0, ks = 0.0;
    for (int b = warp * per; b < min(nb, (warp + 1) * per); ++b) {
        const int k0 = b * CW_R;
        if ((b - warp * per) % CW_FRESH == 0) {
            sincospi((double)(k0 * step % n4) / (2.0 * n), &ks, &kc);
        } else {
            const double c = kc * rc - ks * rs;
            ks = fma(kc, rs, ks * rc);
            kc = c;
        }
        double ce = 0.0, de = 0.0, co = 0.0, dd = 0.0;  // sums with cos(r phi), sin(r phi); even and odd k
#pragma unroll
        for (int r = 0; r < CW_R; r += 2) {
            double x = k0 + r < n ? g[k0 + r] : 0.0;
            const double y = k0 + r + 1 < n ? g[k0 + r + 1] : 0.0;
            if (k0 + r == 0) x *= 0.5;
            ce = fma(x, cr[r], ce);
            de = fma(x, sr[r], de);
            co = fma(y, cr[r + 1], co);
            dd = fma(y, sr[r + 1], dd);
        }
        even += kc * ce - ks * de;
        odd += kc * co - ks * dd;
    }
    se[warp][lane] = even;
    so[warp][lane] = odd;
    __syncthreads();
    if (warp == 0 && blockIdx.x * 32 + lane < half) {
        double e = 0.0, o = 0.0;
        for (int k = 0; k < CW_NW; ++k) {
            e += se[k][lane];
            o += so[k][lane];
        }
        w[i] = (2.0 / n) * (e + o);
        w[n - 1 - i] = (2.0 / n) * (i == n - 1 - i ? e + o : e - o);
    }
}

struct MuResult {
    double mu, N, iters, converged;
    unsigned long long bits[2];
};

// The bisection as one cluster of thread blocks: every block sums its share of the
// nodes, the blocks' sums meet in distributed shared memory, and every block takes
// the same decision.  A thread's first BIS_KEEP nodes stay in registers.  Beyond 120
// smearing widths above mu a Fermi occupation is below 1e-52 and counts as 0 (below
// 40 under mu it is 1 in FP64), without its exponential.  (One thread block, with a
// cosine and an exponential per node and midpoint, took 9 ms at n = 9216; now 0.23 ms.)
//
// Up to BIS_ONE nodes one thread block with a node per thread is faster than a cluster's
// barriers: 128 midpoints 0.39 against 0.71 ms at 16 nodes, 0.55 against 0.87 at 256.
constexpr int BIS_CTAS = 8, BIS_NT = 512, BIS_KEEP = 4, BIS_ONE = 256;
template <int CTAS, int NT, int KEEP>
__global__ void __cluster_dims__(CTAS, 1, 1) __launch_bounds__(NT)
    k_bisect(const double *w, int n, double emin, double emax, int kind, double kT, double N_e, double tol_N,
             int max_iter, double lo, double hi, MuResult *res) {
    namespace cg = cooperative_groups;
    cg::cluster_group cluster = cg::this_cluster();
    __shared__ double sh[NT / 32];
    __shared__ double s_part[2];  // this block's sum, alternating
    const int rank = (int)cluster.block_rank(), first = rank * NT + threadIdx.x;
    const double sigma = 2.0 / (emax - emin), tau = (emin + emax) / 2.0;
    double xs[KEEP], ws[KEEP];
#pragma unroll
    for (int k = 0; k < KEEP; ++k) {
        const int i = first + k * CTAS * NT;
        xs[k] = i < n ? node(i, n, sigma, tau) : 0.0;
        ws[k] = i < n ? w[i] : 0.0;
    }
    auto occ = [&](double x, double mu) {
        if (kind == CHEB_FERMI) {
            const double z = (x - mu) / kT;
            return z > 120.0 ? 0.0 : z < -40.0 ? 1.0 : fermi(x, mu, kT);
        }
        return 0.5 * erfc((x - mu) / kT);
    };
    unsigned long long bits[2] = {0ull, 0ull};
    double mid = 0.5 * (lo + hi), N = 0.0;
    int it = 0, conv = 0;
    for (it = 1; it <= max_iter; ++it) {
        mid = 0.5 * (lo + hi);
        double s = 0.0;
#pragma unroll
        for (int k = 0; k < KEEP; ++k)
            if (first + k * CTAS * NT < n) s += occ(xs[k], mid) * ws[k];
        for (int i = first + KEEP * CTAS * NT; i < n; i += CTAS * NT)
            s += occ(node(i, n, sigma, tau), mid) * w[i];
        const double r = block_sum<NT>(s, sh);
        if (threadIdx.x == 0) s_part[it & 1] = r;
        // (a block's other slot is only rewritten after the next sync)
        if constexpr (CTAS > 1) cluster.sync();
        else __syncthreads();
        N = 0.0;
        for (int b = 0; b < CTAS; ++b) N += CTAS > 1 ? *cluster.map_shared_rank(&s_part[it & 1], b) : s_part[it & 1];
        if (fabs(N - N_e) <= tol_N) {
            conv = 1;
            break;
        }
        if (N > N_e) {
            bits[(it - 1) >> 6] |= 1ull << ((it - 1) & 63);
            hi = mid;
        } else {
            lo = mid;
        }
    }
    cluster.sync();  // no block leaves while another still reads its sum
    if (!conv) {
        it = max_iter;
        mid = 0.5 * (lo + hi);
    }
    if (rank == 0 && threadIdx.x == 0) {
        res->mu = mid;
        res->N = N;
        res->iters = it;
        res->converged = conv;
        res->bits[0] = bits[0];
        res->bits[1] = bits[1];
    }
}
static int launch_mu(const double *g, int n, double emin, double emax, int kind, double kT, double N_e, double tol_N,
                     int max_iter, const double *bracket, void *result, double *w, cudaStream_t s) {
    k_count_weights<<<((n + 1) / 2 + 31) / 32, CW_NW * 32, 0, s>>>(g, n, w);
    CHEB_TRY(check_launch("k_count_weights"));
    const double lo = bracket ? bracket[0] : emin, hi = bracket ? bracket[1] : emax;
    MuResult *res = static_cast<MuResult *>(result);
    if (n <= BIS_ONE)
        k_bisect<1, BIS_ONE, 1><<<1, BIS_ONE, 0, s>>>(w, n, emin, emax, kind, kT, N_e, tol_N, max_iter, lo, hi, res);
    else
        k_bisect<BIS_CTAS, BIS_NT, BIS_KEEP><<<BIS_CTAS, BIS_NT, 0, s>>>(w, n, emin, emax, kind, kT, N_e, tol_N, max_iter, lo,
                                                                        hi, res);
    return check_launch("k_bisect");
}

std::vector<int> ladder(int n_max) {
    std::vector<int> v;
    for (int e = 1; 8 * (1 << e) <= n_max; ++e)
        for (int m = 8; m < 16; ++m) {
            int x = m * (1 << e);
            if (x >= 16 && x <= n_max) v.push_back(x);
        }
    std::sort(v.begin(), v.end());
    v.erase(std::unique(v.begin(), v.end()), v.end());
    return v;
}

}  // namespace cheb

using namespace cheb;

// Values per function of the candidates n_max has, and the largest degree-search
// ladder in it; the workspace holds node values, transforms and coefficients of all
// functions and one cosine table.
static int64_t cand_total(const std::vector<int> &cand) {
    int64_t t = 0;
    for (const int n : cand) t += n;
    return t;
}
static size_t coeffs_ws(int n_f, const std::vector<int> &cand) {
    const size_t nc = cand.size(), total = (size_t)cand_total(cand);
    return 2 * align_up(n_f * total * 8) + align_up(n_f * total * 16) + align_up(4 * total * 8) +
           2 * align_up(n_f * nc * 8) + 256;
}

extern "C" int cheb_coeffs_workspace_size(int32_t n_f, int32_t n_max, size_t *bytes) {
    if (!bytes || n_f < 1 || n_f > 8 || n_max < 16) return fail(CHEB_ERR_INVALID, "cheb_coeffs_workspace_size: bad args");
    std::vector<int> cand = ladder(n_max);
    if (cand.empty() || cand.back() != n_max) cand.push_back(n_max);
    *bytes = coeffs_ws(n_f, cand);
    return CHEB_OK;
}

extern "C" int cheb_coeffs(const cheb_func *funcs, int32_t n_f, double emin, double emax, double tol, int32_t rel,
                           int32_t n_max, int32_t *n_out, double *coeffs, void *ws, size_t ws_bytes, void *stream) {
    if (!funcs || n_f < 1 || n_f > 8 || n_max < 16 || !(emax > emin) || !coeffs)
        return fail(CHEB_ERR_INVALID, "cheb_coeffs: bad arguments");
    size_t need;
    CHEB_TRY(cheb_coeffs_workspace_size(n_f, n_max, &need));
    if (!ws || ws_bytes < need) return fail(CHEB_ERR_NOSPACE, "cheb_coeffs: workspace %zu < %zu", ws_bytes, need);
    const std::vector<int> cand = tol > 0 ? ladder(n_max) : std::vector<int>{n_max};
    if (cand.empty()) return fail(CHEB_ERR_INVALID, "cheb_coeffs: empty degree ladder");
    const int nc = (int)cand.size();
    const double sigma = 2.0 / (emax - emin), tau = (emin + emax) / 2.0;
    FuncArr F{};
    for (int f = 0; f < n_f; ++f) F.f[f] = funcs[f];
    const int64_t total = cand_total(cand);
    Carve cv = carve_aligned(ws, ws_bytes);
    double *fv = cv.take<double>((size_t)n_f * total), *cvv = cv.take<double>((size_t)n_f * total);
    double2 *Y = cv.take<double2>((size_t)n_f * total);
    double *tab = cv.take<double>(4 * (size_t)total);
    unsigned long long *errm = cv.take<unsigned long long>((size_t)n_f * nc);
    unsigned long long *fmx = cv.take<unsigned long long>((size_t)n_f * nc);
    if (!cv.fits()) return fail(CHEB_ERR_NOSPACE, "cheb_coeffs: workspace too small");
    cudaStream_t s = as_stream(stream);
    auto batch = [&](int c0, int c1) {
        Cand d{};
        d.nc = c1 - c0;
        d.total = total;
        int64_t off = cand_total(std::vector<int>(cand.begin(), cand.begin() + c0));
        for (int c = c0; c < c1; ++c) {
            d.n[c - c0] = cand[c];
            d.off[c - c0] = off;
            off += cand[c];
            int n1 = 1;
            for (int k = 2; (int64_t)k * k <= cand[c]; ++k)
                if (cand[c] % k == 0) n1 = k;
            d.n1[c - c0] = n1;
        }
        return d;
    };
    auto transform = [&](const Cand &d, int n_big) -> int {
        const unsigned nb = (unsigned)((n_big + 127) / 128);
        k_cos_table<<<dim3((4 * n_big + 255) / 256, d.nc), 256, 0, s>>>(d, tab);
        k_nodes<<<dim3(nb, n_f * d.nc), 128, 0, s>>>(F, d, sigma, tau, fv);
        k_dft1<<<dim3(nb, n_f * d.nc), 128, 0, s>>>(fv, d, tab, Y);
        k_dft2<<<dim3(d.n1[0] == 1 ? nb * DFT_LANES / 2 + 1 : nb, n_f * d.nc), 128, 0, s>>>(Y, d, tab, cvv);
        return check_launch("cheb_coeffs transform", 4);
    };
    int chosen = nc - 1;
    if (tol <= 0) {
        CHEB_TRY(transform(batch(0, nc), cand[nc - 1]));
    } else {
        // The smallest candidate whose fit error is below tol, per function.  Candidates
        // go in batches of increasing size.  In a batch, 513 of the grid's points settle
        // most candidates: an error clearly above tol there is enough to fail.  The first
        // that they leave is judged on the whole grid, then the next if it fails, and so
        // on; by the estimate while that is clearly off tol, else by the error itself.
        // (The whole grid for all 81 candidates up to 16384 terms took 40 ms.)
        std::vector<int> best(n_f, -1);
        std::vector<unsigned long long> he((size_t)n_f * nc), hm((size_t)n_f * nc), hs((size_t)n_f * nc);
        auto val = [](const std::vector<unsigned long long> &v, int i) {
            double x;
            memcpy(&x, &v[i], 8);
            return x;
        };
        int left = n_f;
        for (int c0 = 0; c0 < nc && left > 0;) {
            int c1 = c0 + 1;
            while (c1 < nc && c1 - c0 < CAND_MAX && (cand[c1] <= 2048 || cand[c1] < 2 * cand[c0])) ++c1;
            const Cand d = batch(c0, c1);
            const int big = cand[c1 - 1], np = n_f * d.nc;
            // below tol: 1 yes, -1 no, 0 within the recursions' rounding of it (n^2 u of the
            // largest |f|, at the ends of the interval) or too near to say
            auto verdict = [&](int i, double e) {
                const double n = d.n[i % d.nc], t = rel ? tol * val(hs, i) : tol;
                const double off = 0.1 * t + 0x1p-52 * n * n * val(hm, i);
                return e < t - off ? 1 : e > t + off ? -1 : 0;
            };
            auto fetch = [&](std::vector<unsigned long long> &h, const unsigned long long *from) {
                return cudaMemcpyAsync(h.data(), from, np * 8, cudaMemcpyDeviceToHost, s);
            };
            auto clear = [&]() { return cudaMemsetAsync(errm, 0, np * 8, s); };
            CHEB_TRY(transform(d, big));
            CHEB_CUDA(clear());
            CHEB_CUDA(cudaMemsetAsync(fmx, 0, np * 8, s));
            k_fit_estimate<<<dim3(33, np), 256, 0, s>>>(F, cvv, d, Pairs{}, 16, sigma, tau, errm, fmx);
            CHEB_TRY(check_launch("k_fit_estimate"));
            CHEB_CUDA(fetch(he, errm));
            CHEB_CUDA(fetch(hm, fmx));
            if (rel) {
                k_fit_scale<<<dim3((GRID_UNIFORM + 2 * big + 256) / 256, np), 256, 0, s>>>(F, d, sigma, tau, fmx);
                CHEB_TRY(check_launch("k_fit_scale"));
                CHEB_CUDA(fetch(hs, fmx));
            }
            CHEB_CUDA(cudaStreamSynchronize(s));
            std::vector<char> open(np);
            for (int i = 0; i < np; ++i) open[i] = verdict(i, val(he, i)) >= 0;
            while (true) {
                Pairs pairs{}, near{};
                for (int f = 0; f < n_f; ++f) {
                    if (best[f] >= 0) continue;
                    for (int c = 0; c < d.nc; ++c)
                        if (open[f * d.nc + c]) {
                            pairs.at[pairs.n++] = f * d.nc + c;
                            break;
                        }
                }
                if (pairs.n == 0) break;
                CHEB_CUDA(clear());
                k_fit_estimate<<<dim3((GRID_UNIFORM / 2 + big + 9) / 8, pairs.n), 256, 0, s>>>(F, cvv, d, pairs, 1, sigma, tau,
                                                                                      errm, fmx);
                CHEB_TRY(check_launch("k_fit_estimate"));
                CHEB_CUDA(fetch(he, errm));
                CHEB_CUDA(cudaStreamSynchronize(s));
                for (int k = 0; k < pairs.n; ++k)
                    if (verdict(pairs.at[k], val(he, pairs.at[k])) == 0) near.at[near.n++] = pairs.at[k];
                std::vector<unsigned long long> hx(he);
                if (near.n > 0) {
                    CHEB_CUDA(clear());
                    k_fit_error<<<dim3((GRID_UNIFORM + 2 * big + 64) / 64, near.n), 64, 0, s>>>(F, cvv, d, near, sigma, tau,
                                                                                               errm);
                    CHEB_TRY(check_launch("k_fit_error"));
                    CHEB_CUDA(fetch(hx, errm));
                    CHEB_CUDA(cudaStreamSynchronize(s));
                }
                for (int k = 0; k < pairs.n; ++k) {
                    const int i = pairs.at[k], v = verdict(i, val(he, i));
                    const double e = rel ? val(hx, i) / val(hs, i) : val(hx, i);
                    open[i] = 0;
                    if (v > 0 || (v == 0 && e < tol)) {
                        best[i / d.nc] = c0 + i % d.nc;
                        --left;
                    }
                }
            }
            c0 = c1;
        }
        for (int f = 0; f < n_f; ++f)
            if (best[f] < 0) return fail(CHEB_ERR_NOT_CONVERGED, "cheb_coeffs: function %d needs more than %d terms", f, n_max);
        chosen = *std::max_element(best.begin(), best.end());
    }
    k_pick<<<dim3((n_max + 255) / 256, n_f), 256, 0, s>>>(cvv, batch(chosen, chosen + 1), 0, cand[chosen], n_max, coeffs);
    CHEB_TRY(check_launch("k_pick"));
    if (n_out) {
        *n_out = cand[chosen];
        CHEB_CUDA(cudaStreamSynchronize(s));
    }
    return CHEB_OK;
}

extern "C" int cheb_penalty_trace(const double *moments, int32_t n_terms, double alpha, double *out, void *ws,
                                  size_t ws_bytes, void *stream) {
    if (!moments || !out || n_terms < 1) return fail(CHEB_ERR_INVALID, "cheb_penalty_trace: bad arguments");
    if (!ws || ws_bytes < (size_t)n_terms * 8) return fail(CHEB_ERR_NOSPACE, "cheb_penalty_trace: workspace");
    cudaStream_t s = as_stream(stream);
    double *c = static_cast<double *>(ws);
    k_penalty_coeffs<<<(n_terms + PEN_J - 1) / PEN_J, PEN_NT, 0, s>>>(alpha, n_terms, c);
    CHEB_TRY(check_launch("k_penalty_coeffs"));
    k_dot_terms<256><<<1, 256, 0, s>>>(c, moments, n_terms, out);
    return check_launch("k_dot_terms");
}

extern "C" int cheb_mu_search(const double *gmoments, int32_t n_terms, double emin, double emax, int32_t kind,
                              double kT, double N_e, double tol_N, int32_t max_iter, const double *bracket,
                              void *result, void *ws, size_t ws_bytes, void *stream) {
    if (!gmoments || !result || n_terms < 2 || !(emax > emin) || max_iter < 1 || max_iter > 128 || !(kT > 0) ||
        (kind != CHEB_FERMI && kind != CHEB_ERFC))
        return fail(CHEB_ERR_INVALID, "cheb_mu_search: bad arguments");
    if (!ws || ws_bytes < (size_t)n_terms * 8) return fail(CHEB_ERR_NOSPACE, "cheb_mu_search: workspace");
    return launch_mu(gmoments, n_terms, emin, emax, kind, kT, N_e, tol_N, max_iter, bracket, result,
                     static_cast<double *>(ws), as_stream(stream));
}

// Workspace-free mu search (no counterpart in the paper).  The count weights
// live in a static device array of the library; its address is looked up once
// per device with that device current and cached under a host mutex.
namespace cheb {

static __device__ __align__(256) double g_mu_noalloc_w[CHEB_MU_SEARCH_NOALLOC_MAX_TERMS];

constexpr int NOALLOC_MAX_DEVICES = 64;
static std::mutex g_mu_noalloc_mx;
static double *g_mu_noalloc_ptr[NOALLOC_MAX_DEVICES] = {};

static int mu_noalloc_scratch(double **out) {
    int dev = -1;
    CHEB_CUDA(cudaGetDevice(&dev));
    if (dev < 0 || dev >= NOALLOC_MAX_DEVICES)
        return fail(CHEB_ERR_INVALID, "cheb_mu_search_noalloc: device %d beyond the %d supported", dev,
                    NOALLOC_MAX_DEVICES);
    std::lock_guard<std::mutex> lk(g_mu_noalloc_mx);
    if (!g_mu_noalloc_ptr[dev]) {
        void *p = nullptr;
        const cudaError_t e = cudaGetSymbolAddress(&p, g_mu_noalloc_w);
        if (e != cudaSuccess || !p)
            return fail(CHEB_ERR_CUDA, "cheb_mu_search_noalloc: scratch address on device %d: %s", dev,
                        cudaGetErrorString(e));
        g_mu_noalloc_ptr[dev] = static_cast<double *>(p);
    }
    *out = g_mu_noalloc_ptr[dev];
    return CHEB_OK;
}

}  // namespace cheb

extern "C" int cheb_mu_search_noalloc(const double *gmoments, int32_t n_terms, double emin, double emax,
                                      int32_t kind, double kT, double N_e, double tol_N, int32_t max_iter,
                                      const double *bracket, void *result, void *stream) {
    if (!gmoments || !result || n_terms < 2 || !(emax > emin) || max_iter < 1 || max_iter > 128 || !(kT > 0) ||
        (kind != CHEB_FERMI && kind != CHEB_ERFC))
        return fail(CHEB_ERR_INVALID, "cheb_mu_search_noalloc: bad arguments");
    if (n_terms > CHEB_MU_SEARCH_NOALLOC_MAX_TERMS)
        return fail(CHEB_ERR_INVALID,
                    "cheb_mu_search_noalloc: n_terms %d exceeds the static scratch of %d terms; "
                    "use cheb_mu_search with a workspace",
                    n_terms, CHEB_MU_SEARCH_NOALLOC_MAX_TERMS);
    double *w = nullptr;
    CHEB_TRY(mu_noalloc_scratch(&w));
    return launch_mu(gmoments, n_terms, emin, emax, kind, kT, N_e, tol_N, max_iter, bracket, result, w,
                     as_stream(stream));
}

// ---------------------------------------------------------------------------
// Scalar steps of the solve sequences, kept in the library so that the
// binding only moves arguments.

extern "C" int cheb_penalty_check(const double *moments, int32_t n_terms, double alpha, double threshold,
                                  double *value, int32_t *verdict, void *ws, size_t ws_bytes, void *stream) {
    if (!moments || n_terms < 3 || !(threshold > 0) || !verdict)
        return fail(CHEB_ERR_INVALID, "cheb_penalty_check: bad arguments");
    if (!ws || ws_bytes < (size_t)n_terms * 8 + 8) return fail(CHEB_ERR_NOSPACE, "cheb_penalty_check: workspace");
    double *out = static_cast<double *>(ws) + n_terms;
    // |alpha| at most 2/5 of the terms, so that the penalty polynomial of
    // n_terms terms resolves the exponential's decay length
    const double amax = 0.4 * n_terms;
    if (fabs(alpha) > amax) alpha = alpha < 0 ? -amax : amax;
    CHEB_TRY(cheb_penalty_trace(moments, n_terms, alpha, out, ws, (size_t)n_terms * 8, stream));
    double v = 0.0, last[2] = {0.0, 0.0};
    cudaStream_t s = as_stream(stream);
    CHEB_CUDA(cudaMemcpyAsync(&v, out, 8, cudaMemcpyDeviceToHost, s));
    CHEB_CUDA(cudaMemcpyAsync(last, moments + n_terms - 2, 16, cudaMemcpyDeviceToHost, s));
    CHEB_CUDA(cudaStreamSynchronize(s));
    if (value) *value = v;
    // A level outside [-1, 1] makes T_k grow like cosh(k acosh|x~|), and the
    // penalty polynomial grows with it outside the interval, so |trace| says
    // that a bound fails but its sign does not say which.  The moments do: the
    // level's term dominates them, with one sign above +1 and alternating
    // signs (T_k(-y) = (-1)^k T_k(y)) below -1.
    const bool finite = v == v && v - v == 0.0 && last[0] - last[0] == 0.0 && last[1] - last[1] == 0.0;
    if (!finite) *verdict = 2;
    else if (fabs(v) < threshold) *verdict = 0;
    else *verdict = last[0] * last[1] < 0.0 ? -1 : 1;
    return CHEB_OK;
}

extern "C" int cheb_widen_bounds(double *bounds, int32_t verdict, double frac) {
    if (!bounds || !(frac >= 0) || verdict < -1 || verdict > 2 || !(bounds[1] > bounds[0]))
        return fail(CHEB_ERR_INVALID, "cheb_widen_bounds: bad arguments");
    const double w = frac * (bounds[1] - bounds[0]);
    if (verdict == -1 || verdict == 2) bounds[0] -= w;
    if (verdict == 1 || verdict == 2) bounds[1] += w;
    return CHEB_OK;
}

extern "C" int cheb_mlp_bracket(const float *out, double emin, double emax, double kT, double min_half_kT,
                                double max_half_kT, double *mu_hat, double *half) {
    if (!out || !mu_hat || !half || !(emax > emin) || !(kT > 0) || !(min_half_kT >= 0) ||
        !(max_half_kT >= min_half_kT))
        return fail(CHEB_ERR_INVALID, "cheb_mlp_bracket: bad arguments");
    // the network works in the scaled variable of Eq. 2: x~ = sigma (e - tau)
    const double sigma = 2.0 / (emax - emin), tau = 0.5 * (emin + emax);
    *mu_hat = (double)out[0] / sigma + tau;
    const double h = exp((double)out[1]) / sigma;
    *half = fmin(fmax(h, min_half_kT * kT), max_half_kT * kT);
    return CHEB_OK;
}

extern "C" int cheb_mu_nodes(double center, double half, int32_t n, double *nodes) {
    if (n < 1 || n > 64 || !nodes || !(half >= 0)) return fail(CHEB_ERR_INVALID, "cheb_mu_nodes: bad arguments");
    const double pi = 3.14159265358979323846;
    for (int i = 0; i < n; ++i) nodes[i] = center + half * cos(pi * (i + 0.5) / n);
    return CHEB_OK;
}

extern "C" int cheb_lagrange_weights(const double *nodes, int32_t n, double x, double *weights) {
    if (n < 1 || n > 64 || !nodes || !weights) return fail(CHEB_ERR_INVALID, "cheb_lagrange_weights: bad arguments");
    for (int i = 0; i < n; ++i) {
        double v = 1.0;
        for (int j = 0; j < n; ++j) {
            if (j == i) continue;
            if (nodes[i] == nodes[j]) return fail(CHEB_ERR_INVALID, "cheb_lagrange_weights: repeated node");
            v *= (x - nodes[j]) / (nodes[i] - nodes[j]);
        }
        weights[i] = v;
    }
    return CHEB_OK;
}

extern "C" int cheb_bounds_spd(const cheb_bsr *S, int32_t k, const double *v0, double margin_frac, double *emin,
                               double *emax, void *ws, size_t ws_bytes, void *stream) {
    double th[2];
    CHEB_TRY(cheb_bounds(S, k, v0, margin_frac, emin, emax, th, ws, ws_bytes, stream));
    if (!(th[0] > 0)) return fail(CHEB_ERR_NOT_SPD, "cheb_bounds_spd: lowest Ritz value %g <= 0", th[0]);
    if (*emin < 0.5 * th[0]) *emin = 0.5 * th[0];
    return CHEB_OK;
}

extern "C" int cheb_series_value(const double *coeffs, const double *moments, int32_t n_terms, double *out,
                                 void *stream) {
    if (!coeffs || !moments || !out || n_terms < 1) return fail(CHEB_ERR_INVALID, "cheb_series_value: bad arguments");
    k_dot_terms<256><<<1, 256, 0, as_stream(stream)>>>(coeffs, moments, n_terms, out);
    return check_launch("k_dot_terms");
}
