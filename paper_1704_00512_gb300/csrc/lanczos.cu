// Spectral bounds from a few Lanczos steps (Sec. "Determination of the
// eigenvalue bounds and polynomial degree" suggests "a few steps of a Lanczos
// method" when no earlier bounds exist).  Plain Lanczos without
// reorthogonalisation on the FP64 block-sparse matrix, all reductions in a
// fixed order; then, in one thread block, the extreme eigenvalues of the tridiagonal
// by Sturm-sequence multisection and the last component of their eigenvectors by
// inverse iteration (tridiagonal solve with partial pivoting).
#include <algorithm>
#include <cmath>

#include "common.cuh"

namespace cheb {

constexpr int LZ_GRID = 456;  // thread blocks of the product (three per SM), and at most of the others
constexpr int LZ_NT = 256;

struct LzState {
    double alpha[512];
    double beta[512];
    double partial[2][LZ_GRID];
    double out[8];  // emin, emax, theta_min, theta_max, res_lo, res_hi
    int kk;         // steps actually taken (a breakdown stops early)
};

// The sum of one set of partials, in a fixed order, in every thread.  Every block of
// the kernel that needs it takes it anew: a few hundred values from L2 cost less than a launch
// of their own.
__device__ __forceinline__ double lz_total(const double *partial, int np, double *sh) {
    double s = 0.0;
    for (int i = threadIdx.x; i < np; i += LZ_NT) s += partial[i];
    const double r = block_sum<LZ_NT>(s, sh);
    if (threadIdx.x == 0) sh[0] = r;
    __syncthreads();
    const double t = sh[0];
    __syncthreads();
    return t;
}

// A Lanczos step is three kernels; each also finishes the sum that the one before
// left in parts.  (Six launches a step, among them two of one block, and a product
// whose lanes each read a 128-byte block by itself took 117 us a step at 20,000
// rows; now about 45 us.)
//
// 1: w = A v - beta_{j-1} v_{j-1}, and the parts of alpha_j = w.v.  One warp per block
// row; a row's values are one stream, a double2 per lane: lane l has row (l / 2) % 4
// of every fourth block and columns 2 (l % 2), + 1, and 32 blocks are on their
// way, the next ones' columns too.  Neighbouring rows go to different SMs: what
// bounds it is the FP64 pipe (18 us at 20,000 rows and 144 blocks a row), and an SM with
// a block of rows more than others makes all wait.  (wide: the values are aligned
// for that; else two doubles.)
__device__ __forceinline__ double2 lz_pair(const double *p, int wide) {
    return wide ? __ldg(reinterpret_cast<const double2 *>(p)) : make_double2(__ldg(p), __ldg(p + 1));
}
__global__ void __launch_bounds__(LZ_NT, 3) k_lz_product(const int64_t *rp, const int32_t *ci, const double *a, int64_t nbr,
                                                      const double *v, const double *vm, double *w, LzState *st, int step, int wide) {
    if (step >= st->kk) return;
    __shared__ double sh[LZ_NT / 32];
    const int lane = threadIdx.x & 31, r = (lane >> 1) & 3;
    const double beta = step > 0 ? st->beta[step - 1] : 0.0;
    double s = 0.0;
    for (int64_t I = blockIdx.x + (int64_t)gridDim.x * (threadIdx.x >> 5); I < nbr; I += ((int64_t)gridDim.x * LZ_NT) >> 5) {
        const int64_t b1 = rp[I + 1];
        int64_t b0 = rp[I];
        double acc = 0.0, acc2 = 0.0;
        int col = b0 + lane < b1 ? ci[b0 + lane] : 0;
        for (; b0 < b1; b0 += 32) {
            double2 m[8];
            int64_t k[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int64_t b = b0 + 4 * u + (lane >> 3);
                m[u] = b < b1 ? lz_pair(a + b * BB + 2 * (lane & 7), wide) : make_double2(0.0, 0.0);
                k[u] = (int64_t)__shfl_sync(0xffffffffu, col, 4 * u + (lane >> 3)) * BS + 2 * (lane & 1);
            }
            col = b0 + 32 + lane < b1 ? ci[b0 + 32 + lane] : 0;
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                if (b0 + 4 * u + (lane >> 3) < b1) {
                    const double2 x = *reinterpret_cast<const double2 *>(v + k[u]);
                    if (u & 1) acc2 = fma(m[u].x, x.x, fma(m[u].y, x.y, acc2));
                    else acc = fma(m[u].x, x.x, fma(m[u].y, x.y, acc));
                }
            }
        }
        acc += acc2;
        acc += __shfl_xor_sync(0xffffffffu, acc, 1);
        acc += __shfl_xor_sync(0xffffffffu, acc, 8);
        acc += __shfl_xor_sync(0xffffffffu, acc, 16);
        if ((lane & 25) == 0) {
            const int64_t i = I * BS + r;
            const double x = acc - beta * vm[i];
            w[i] = x;
            s += x * v[i];
        }
    }
    const double t = block_sum<LZ_NT>(s, sh);
    if (threadIdx.x == 0) st->partial[0][blockIdx.x] = t;
}

// 2: alpha_j; w -= alpha_j v, and the parts of w.w.  (start: the parts of w.w alone.)
__global__ void __launch_bounds__(LZ_NT) k_lz_alpha(int start, int64_t n, double *w, const double *v, LzState *st, int step) {
    if (step >= st->kk) return;
    __shared__ double sh[LZ_NT / 32];
    const double alpha = start ? 0.0 : lz_total(st->partial[0], LZ_GRID, sh);
    double s = 0.0;
    for (int64_t i = blockIdx.x * (int64_t)LZ_NT + threadIdx.x; i < n; i += (int64_t)gridDim.x * LZ_NT) {
        double x = w[i];
        if (!start) {
            x = x - alpha * v[i];
            w[i] = x;
        }
        s += x * x;
    }
    const double r = block_sum<LZ_NT>(s, sh);
    if (threadIdx.x == 0) st->partial[1][blockIdx.x] = r;
    if (!start && blockIdx.x == 0 && threadIdx.x == 0) st->alpha[step] = alpha;
}

// 3: beta_j = |w|; v_{j-1} = v, v = w / beta_j -- unless the step is a breakdown: a beta
// at rounding level of the step's scale means that the Krylov space is invariant
// (e.g. a multiple of the identity), and later steps would only amplify rounding
// noise.  (start: v = w / |w|, v_{j-1} = 0.)
__global__ void __launch_bounds__(LZ_NT) k_lz_next(int start, int64_t n, const double *w, double *v, double *vm, LzState *st,
                                                   int step) {
    if (step >= st->kk) return;
    __shared__ double sh[LZ_NT / 32];
    const double b = sqrt(lz_total(st->partial[1], gridDim.x, sh));
    if (!start) {
        const double ref = fabs(st->alpha[step]) + (step > 0 ? st->beta[step - 1] : 0.0);
        const bool stop = b == 0.0 || b <= 1e-12 * ref;
        if (blockIdx.x == 0 && threadIdx.x == 0) st->beta[step] = b;
        if (stop) {  // (every block finds the same)
            if (blockIdx.x == 0 && threadIdx.x == 0) st->kk = step + 1;
            return;
        }
    }
    for (int64_t i = blockIdx.x * (int64_t)LZ_NT + threadIdx.x; i < n; i += (int64_t)gridDim.x * LZ_NT) {
        vm[i] = start ? 0.0 : v[i];
        v[i] = w[i] / b;
    }
}

// The default start vector: x_i = 1 + u_i / 2, u_i = (splitmix64(i) >> 11) / 2^53
// (SplitMix64: Steele, Lea and Flood, 2014).  Positive like the all-ones
// vector, but with a component along every eigenvector of a structured matrix
// (the all-ones vector can lie in a small invariant subspace, e.g. of the
// overlap of one atom's basis functions, and Lanczos would then stop inside it).
__device__ __forceinline__ uint64_t lz_splitmix64(uint64_t x) {
    uint64_t z = x + 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}
__global__ void k_fill_start(double *x, int64_t n) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        x[i] = 1.0 + 0.5 * ((double)(lz_splitmix64((uint64_t)i) >> 11) * (1.0 / 9007199254740992.0));
}

// Number of eigenvalues of the tridiagonal (a, b) below x: the sign changes of the
// leading minors p_i = (a_i - x) p_{i-1} - b_{i-1}^2 p_{i-2} (Sturm sequence; a zero
// counts with the sign before it).  |a|, |b| <= 1: eight steps stay in range, then the
// pair is scaled by a power of two.  (The quotients p_i / p_{i-1} need no scaling, but
// a division each, ten dependent FP64 operations.)
__device__ int sturm_count(const double *a, const double *b2, int k, double x) {
    double pm = 1.0, p = a[0] - x;
    bool neg = p < 0.0;
    int c = neg;
    for (int i = 1; i < k; ++i) {
        const double q = fma(a[i] - x, p, -b2[i - 1] * pm);
        pm = p;
        p = q;
        const bool n = q < 0.0 || (q == 0.0 && neg);
        c += n != neg;
        neg = n;
        if ((i & 7) == 0) {
            const int e = max(__double2hiint(p) & 0x7ff00000, __double2hiint(pm) & 0x7ff00000);
            if (e > 0x00200000 && e < 0x7fc00000) {
                const double f = __hiloint2double(0x7fe00000 - e, 0);
                p *= f;
                pm *= f;
            }
        }
    }
    return c;
}

// Last component of the unit eigenvector for eigenvalue th: inverse iteration, three
// solves of (T - th I) y = y_prev with one factorisation by Gaussian elimination with
// partial pivoting.  f: multipliers, rd: reciprocals of the pivots, du: superdiagonal
// (a pivoted row i has b[i + 1] beyond it).  |a|, |b| <= 1.
__device__ double last_component(const double *a, const double *b, int k, double th, double *f, double *rd, double *du,
                                 double *y, unsigned char *piv) {
    if (k == 1) return 1.0;
    // the place of a pivot that is zero (th an eigenvalue to the last bit): small enough to
    // leave the eigenvector alone, large enough for the squares of what it gives
    constexpr double tiny = 1e-100;
    double d = a[0] - th, u = b[0];
    for (int i = 0; i < k - 1; ++i) {
        double dn = a[i + 1] - th, un = i < k - 2 ? b[i + 1] : 0.0;
        const bool p = fabs(d) < fabs(b[i]);
        if (!p && d == 0.0) d = tiny;
        rd[i] = 1.0 / (p ? b[i] : d);
        const double m = (p ? d : b[i]) * rd[i];
        if (p) {
            du[i] = dn;
            dn = u - m * dn;
            un = -m * un;
        } else {
            du[i] = u;
            dn -= m * u;
        }
        f[i] = m;
        piv[i] = p;
        d = dn;
        u = un;
    }
    rd[k - 1] = 1.0 / (d == 0.0 ? tiny : d);
    for (int i = 0; i < k; ++i) y[i] = 1.0;
    for (int it = 0; it < 3; ++it) {
        double cur = y[0];
        for (int i = 0; i < k - 1; ++i) {
            const double nx = y[i + 1], m = f[i];
            const bool p = piv[i];
            y[i] = p ? nx : cur;
            cur = p ? cur - m * nx : nx - m * cur;
        }
        double y1 = cur * rd[k - 1], y2 = 0.0, nrm = y1 * y1;
        y[k - 1] = y1;
        for (int i = k - 2; i >= 0; --i) {
            const double w = piv[i] && i < k - 2 ? b[i + 1] * y2 : 0.0;
            y2 = y1;
            y1 = (y[i] - w - du[i] * y1) * rd[i];
            y[i] = y1;
            nrm = fma(y1, y1, nrm);
        }
        nrm = 1.0 / sqrt(nrm);
        for (int i = 0; i < k; ++i) y[i] *= nrm;
    }
    return y[k - 1];
}

// The extreme eigenvalues and the last components of their eigenvectors: warp 0 the
// lowest, warp 1 the highest, each by multisection of the Gershgorin interval, a Sturm
// count per lane (33 parts a round: 11 rounds instead of 55 halvings; more lanes would
// be bound by the FP64 pipe).  The matrix is scaled by a power of two.  (One thread for
// all of it, its vectors in global memory, took 1.2 ms at k = 40; now 0.16 ms.)
__global__ void __launch_bounds__(64) k_tridiag(LzState *st, double margin_frac) {
    __shared__ double th[2], last[2], ab[3][512], scratch[2][4][512];
    __shared__ unsigned char piv[2][512];
    const int k = st->kk, lane = threadIdx.x & 31, which = threadIdx.x >> 5;
    double lo = st->alpha[0], hi = lo;
    for (int i = 0; i < k; ++i) {
        const double r = (i > 0 ? fabs(st->beta[i - 1]) : 0.0) + (i < k - 1 ? fabs(st->beta[i]) : 0.0);
        lo = fmin(lo, st->alpha[i] - r);
        hi = fmax(hi, st->alpha[i] + r);
    }
    const double big = fmax(fabs(lo), fabs(hi));
    int e = 0;
    if (big > 0.0 && isfinite(big)) frexp(big, &e);
    lo = ldexp(lo, -e);  // (2^-e need not be a double itself)
    hi = ldexp(hi, -e);
    for (int i = threadIdx.x; i < k; i += 64) {
        ab[0][i] = ldexp(st->alpha[i], -e);
        ab[1][i] = ldexp(st->beta[i], -e);
        ab[2][i] = ab[1][i] * ab[1][i];
    }
    __syncthreads();
    const double *a = ab[0], *b = ab[1], *b2 = ab[2];
    {
        double l = lo, h = hi;
        const int target = which == 0 ? 1 : k;
        for (int it = 0; it < 200; ++it) {
            const double m = fmin(h, l + (h - l) * ((lane + 1) / 33.0));
            const bool in = m > l && m < h;
            const bool above = in && sturm_count(a, b2, k, m) >= target;
            const unsigned any = __ballot_sync(0xffffffffu, in), up = __ballot_sync(0xffffffffu, above);
            if (!any) {
                // the interval is a few ulps wide: halve it
                const double c = 0.5 * (l + h);
                if (!(c > l && c < h)) break;
                if (sturm_count(a, b2, k, c) >= target) h = c; else l = c;
                continue;
            }
            // (the counts rise with m: the first point above ends the interval, the last
            // point below starts it)
            const unsigned below = any & ~up;
            const double nh = up ? __shfl_sync(0xffffffffu, m, __ffs(up) - 1) : h;
            const unsigned bl = up ? below & ((1u << (__ffs(up) - 1)) - 1u) : below;
            if (bl) l = __shfl_sync(0xffffffffu, m, 31 - __clz(bl));
            h = nh;
        }
        if (lane == 0) {
            const double t = which == 0 ? h : l;
            th[which] = ldexp(t, e);
            last[which] = last_component(a, b, k, t, scratch[which][0], scratch[which][1], scratch[which][2],
                                         scratch[which][3], piv[which]);
        }
    }
    __syncthreads();
    if (threadIdx.x != 0) return;
    const double bl = st->beta[k - 1];
    const double slo = last[0], shi = last[1];
    const double rlo = fabs(bl * slo), rhi = fabs(bl * shi);
    const double width = th[1] - th[0];
    const double mlo = fmax(2.0 * rlo, margin_frac * width), mhi = fmax(2.0 * rhi, margin_frac * width);
    double e0 = th[0] - mlo, e1 = th[1] + mhi;
    // a (near-)degenerate spectrum still gets an interval to scale by: at
    // least 1e-3 of its magnitude (1e-3 around zero), centred on the Ritz values
    const double mag = fmax(fabs(th[0]), fabs(th[1]));
    const double wmin = 1e-3 * (mag > 0.0 ? mag : 1.0);
    if (e1 - e0 < wmin) {
        const double c = 0.5 * (th[0] + th[1]);
        e0 = fmin(e0, c - 0.5 * wmin);
        e1 = fmax(e1, c + 0.5 * wmin);
    }
    st->out[0] = e0;
    st->out[1] = e1;
    st->out[2] = th[0];
    st->out[3] = th[1];
    st->out[4] = rlo;
    st->out[5] = rhi;
}

}  // namespace cheb

using namespace cheb;

extern "C" int cheb_bounds_workspace_size(int64_t nbr, int32_t k, size_t *bytes) {
    if (!bytes || nbr < 1 || k < 1 || k > 512) return fail(CHEB_ERR_INVALID, "cheb_bounds_workspace_size: bad args");
    *bytes = 3 * align_up(nbr * BS * 8) + align_up(sizeof(LzState)) + 256;
    return CHEB_OK;
}

extern "C" int cheb_bounds(const cheb_bsr *M, int32_t k, const double *v0, double margin_frac, double *emin,
                           double *emax, double *theta, void *ws, size_t ws_bytes, void *stream) {
    if (!M || !M->vals || M->dtype != CHEB_F64 || M->nbr < 1 || !emin || !emax)
        return fail(CHEB_ERR_INVALID, "cheb_bounds: bad arguments");
    size_t need;
    CHEB_TRY(cheb_bounds_workspace_size(M->nbr, k, &need));
    if (!ws || ws_bytes < need) return fail(CHEB_ERR_NOSPACE, "cheb_bounds: workspace %zu < %zu", ws_bytes, need);
    const int64_t n = M->nbr * BS;
    Carve cv = carve_aligned(ws, ws_bytes);
    double *vm = cv.take<double>(n), *v = cv.take<double>(n), *w = cv.take<double>(n);
    LzState *st = cv.take<LzState>(1);
    if (!cv.fits()) return fail(CHEB_ERR_NOSPACE, "cheb_bounds: workspace %zu too small", ws_bytes);
    cudaStream_t s = as_stream(stream);
    CHEB_CUDA(cudaMemsetAsync(st, 0, sizeof(LzState), s));
    const int kk = k;
    CHEB_CUDA(cudaMemcpyAsync(&st->kk, &kk, sizeof(int), cudaMemcpyHostToDevice, s));
    // start vector (copied so v0 stays untouched) and its normalisation
    if (v0) CHEB_CUDA(cudaMemcpyAsync(w, v0, n * 8, cudaMemcpyDeviceToDevice, s));
    else {
        k_fill_start<<<LZ_GRID, LZ_NT, 0, s>>>(w, n);
        CHEB_TRY(check_launch("k_fill_start"));
    }
    // (both kernels on the same grid: the second sums the first's parts)
    const unsigned grid = (unsigned)std::min<int64_t>(LZ_GRID, (n + LZ_NT - 1) / LZ_NT);
    k_lz_alpha<<<grid, LZ_NT, 0, s>>>(1, n, w, v, st, 0);
    k_lz_next<<<grid, LZ_NT, 0, s>>>(1, n, w, v, vm, st, 0);
    CHEB_TRY(check_launch("lanczos start", 2));
    const int wide = reinterpret_cast<uintptr_t>(M->vals) % 16 == 0;
    for (int j = 0; j < k; ++j) {
        k_lz_product<<<LZ_GRID, LZ_NT, 0, s>>>(M->row_ptr, M->col_idx, (const double *)M->vals, M->nbr, v, vm, w, st, j, wide);
        k_lz_alpha<<<grid, LZ_NT, 0, s>>>(0, n, w, v, st, j);
        k_lz_next<<<grid, LZ_NT, 0, s>>>(0, n, w, v, vm, st, j);
        CHEB_TRY(check_launch("lanczos step", 3));
    }
    k_tridiag<<<1, 64, 0, s>>>(st, margin_frac);
    CHEB_TRY(check_launch("k_tridiag"));
    double out[8];
    CHEB_CUDA(cudaMemcpyAsync(out, st->out, sizeof(out), cudaMemcpyDeviceToHost, s));
    CHEB_CUDA(cudaStreamSynchronize(s));
    *emin = out[0];
    *emax = out[1];
    if (theta) {
        theta[0] = out[2];
        theta[1] = out[3];
    }
    return CHEB_OK;
}

extern "C" int cheb_bounds_warm(const cheb_bsr *M, int32_t k, const double *v0, double margin_frac,
                                const double *warm, double *emin, double *emax, double *theta, void *ws,
                                size_t ws_bytes, void *stream) {
    if (!warm || !(warm[0] < warm[1])) return fail(CHEB_ERR_INVALID, "cheb_bounds_warm: warm interval needs lo < hi");
    CHEB_TRY(cheb_bounds(M, k, v0, margin_frac, emin, emax, theta, ws, ws_bytes, stream));
    // Ritz values lie inside the spectrum: a warm interval that misses the
    // Lanczos interval is provably too narrow there and is extended to it
    *emin = std::fmin(*emin, warm[0]);
    *emax = std::fmax(*emax, warm[1]);
    return CHEB_OK;
}
