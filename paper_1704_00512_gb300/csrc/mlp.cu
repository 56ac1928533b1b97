// Learned mu proposal (not in the paper): a 35 -> 128 -> 128 -> 2 ReLU network
// in FP32 with hand-written forward, loss, backward and Adam kernels.
//
// Parameters are one flat vector: W1[128][35], b1[128], W2[128][128], b2[128],
// W3[2][128], b3[2] (row-major, y = W x + b).  Every reduction runs in a fixed order
// (no atomics), so results are reproducible.
//
// At the training sets' few hundred samples everything is latency: what counts is how
// many launches a step takes and how long the chain of dependent loads in each is.  So
// a thread block takes four samples through all layers, a weight feeds all four, and
// the sums over the batch are split over eight threads.  (A launch per layer, with one
// serial loop per thread, took 233 us for a step at batch 346; now 58 us, of which the
// device works 26.)
#include "common.cuh"

namespace cheb {

constexpr int MLP_IN = 35, MLP_H = 128, MLP_OUT = 2;
constexpr int OFF_W1 = 0, OFF_B1 = OFF_W1 + MLP_H * MLP_IN, OFF_W2 = OFF_B1 + MLP_H,
              OFF_B2 = OFF_W2 + MLP_H * MLP_H, OFF_W3 = OFF_B2 + MLP_H, OFF_B3 = OFF_W3 + MLP_OUT * MLP_H,
              MLP_NPARAMS = OFF_B3 + MLP_OUT;

constexpr int MLP_S = 4, MLP_NT = 512;  // samples and threads of a block

// Rows o = warp, warp + 16, ... of y = W x + b for MLP_S samples (x = relu(xs) when
// relu_in), a warp per row: the row's weights are one coalesced read, and four sums
// over the lanes meet in six shuffles (lanes 8 s ... 8 s + 7 end with sample s).
template <int NIN>
__device__ __forceinline__ void dense_rows(const float *__restrict__ W, const float *__restrict__ b, int nout,
                                           const float (*xs)[MLP_H], bool relu_in, float (*ys)[MLP_H]) {
    constexpr int K = (NIN + 31) / 32;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    float x[MLP_S][K];
#pragma unroll
    for (int s = 0; s < MLP_S; ++s)
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const int i = lane + 32 * k;
            x[s][k] = i < NIN ? xs[s][i] : 0.f;
            if (relu_in) x[s][k] = fmaxf(x[s][k], 0.f);
        }
#pragma unroll 8
    for (int o = warp; o < nout; o += MLP_NT / 32) {
        float v[MLP_S] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const int i = lane + 32 * k;
            const float w = i < NIN ? W[o * NIN + i] : 0.f;
#pragma unroll
            for (int s = 0; s < MLP_S; ++s) v[s] = fmaf(w, x[s][k], v[s]);
        }
        const bool h16 = lane & 16, h8 = lane & 8;
        const float p0 = (h16 ? v[2] : v[0]) + __shfl_xor_sync(0xffffffffu, h16 ? v[0] : v[2], 16);
        const float p1 = (h16 ? v[3] : v[1]) + __shfl_xor_sync(0xffffffffu, h16 ? v[1] : v[3], 16);
        float r = (h8 ? p1 : p0) + __shfl_xor_sync(0xffffffffu, h8 ? p0 : p1, 8);
        r += __shfl_xor_sync(0xffffffffu, r, 4);
        r += __shfl_xor_sync(0xffffffffu, r, 2);
        r += __shfl_xor_sync(0xffffffffu, r, 1);
        if ((lane & 7) == 0) ys[lane >> 3][o] = r + b[o];
    }
}

// All three layers; act keeps the pre-activations of the hidden ones, a1 then a2.
__global__ void __launch_bounds__(MLP_NT) k_mlp_forward(const float *__restrict__ theta, const float *__restrict__ X,
                                                        int B, float *__restrict__ act, float *__restrict__ out) {
    __shared__ float x[MLP_S][MLP_H], h1[MLP_S][MLP_H], h2[MLP_S][MLP_H], y[MLP_S][MLP_H];
    const int64_t s0 = (int64_t)blockIdx.x * MLP_S;
    const int s = threadIdx.x / MLP_H, i = threadIdx.x % MLP_H;
    const bool in = s0 + s < B;
    x[s][i] = in && i < MLP_IN ? X[(s0 + s) * MLP_IN + i] : 0.f;
    __syncthreads();
    dense_rows<MLP_IN>(theta + OFF_W1, theta + OFF_B1, MLP_H, x, false, h1);
    __syncthreads();
    if (in) act[(s0 + s) * MLP_H + i] = h1[s][i];
    dense_rows<MLP_H>(theta + OFF_W2, theta + OFF_B2, MLP_H, h1, true, h2);
    __syncthreads();
    if (in) act[(B + s0 + s) * MLP_H + i] = h2[s][i];
    dense_rows<MLP_H>(theta + OFF_W3, theta + OFF_B3, MLP_OUT, h2, true, y);
    __syncthreads();
    if (in && i < MLP_OUT) out[(s0 + s) * MLP_OUT + i] = y[s][i];
}

// Loss of the module docstring of the oracle: d = (xhat - xstar)/scale,
// w = exp(z)/scale, L = huber(d) + relu(|d| - w) + 0.01 w; mean over the batch.
__global__ void k_mlp_loss(const float *out, const float *xstar, const float *scale, int B, float *dout,
                           double *loss) {
    __shared__ double sh[8];
    double acc = 0.0;
    for (int s = threadIdx.x; s < B; s += blockDim.x) {
        const float sc = scale[s];
        const float d = (out[2 * s] - xstar[s]) / sc;
        const float w = expf(out[2 * s + 1]) / sc;
        const float ad = fabsf(d);
        const float hub = ad <= 1.f ? 0.5f * d * d : ad - 0.5f;
        const bool miss = ad > w;
        acc += (double)(hub + (miss ? ad - w : 0.f) + 0.01f * w);
        const float sgn = d > 0.f ? 1.f : (d < 0.f ? -1.f : 0.f);
        const float dh = ad <= 1.f ? d : sgn;
        dout[2 * s] = (dh + (miss ? sgn : 0.f)) / sc / (float)B;
        dout[2 * s + 1] = ((miss ? -1.f : 0.f) + 0.01f) * w / (float)B;
    }
    double r = block_sum<256>(acc, sh);
    if (threadIdx.x == 0 && loss) *loss = r / B;
}

// d2 = (dout W3) [a2 > 0] and d1 = (d2 W2) [a1 > 0], MLP_S samples per block; the sum
// over the 128 rows of W2 is split over four threads.
__global__ void __launch_bounds__(MLP_NT) k_mlp_back(const float *__restrict__ theta, const float *__restrict__ dout,
                                                     const float *__restrict__ a1, const float *__restrict__ a2, int B,
                                                     float *__restrict__ d1, float *__restrict__ d2) {
    __shared__ float4 sd[MLP_H];  // d2 of the four samples
    __shared__ float part[MLP_S][MLP_S][MLP_H];
    static_assert(MLP_S == 4 && MLP_NT == MLP_S * MLP_H, "a thread per sample and unit; as many parts as samples");
    const int64_t s0 = (int64_t)blockIdx.x * MLP_S;
    const int q = threadIdx.x / MLP_H, i = threadIdx.x % MLP_H;  // q: the sample, or the part of the sum
    const bool in = s0 + q < B;
    const size_t at = (s0 + q) * MLP_H + i;
    const float *W2 = theta + OFF_W2 + i, *W3 = theta + OFF_W3 + i;
    float w[MLP_H / MLP_S];
#pragma unroll
    for (int o = 0; o < MLP_H / MLP_S; ++o) w[o] = W2[(q * (MLP_H / MLP_S) + o) * MLP_H];
    float acc = 0.f;
    if (in) {
        acc = fmaf(dout[(s0 + q) * MLP_OUT], W3[0], acc);
        acc = fmaf(dout[(s0 + q) * MLP_OUT + 1], W3[MLP_H], acc);
        acc = a2[at] > 0.f ? acc : 0.f;
        d2[at] = acc;
    }
    reinterpret_cast<float *>(&sd[i])[q] = acc;
    __syncthreads();
    float v[MLP_S] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int o = 0; o < MLP_H / MLP_S; ++o) {
        const float4 d = sd[q * (MLP_H / MLP_S) + o];
        v[0] = fmaf(d.x, w[o], v[0]);
        v[1] = fmaf(d.y, w[o], v[1]);
        v[2] = fmaf(d.z, w[o], v[2]);
        v[3] = fmaf(d.w, w[o], v[3]);
    }
#pragma unroll
    for (int s = 0; s < MLP_S; ++s) part[s][q][i] = v[s];
    __syncthreads();
    if (in) {
        const float r = (part[q][0][i] + part[q][1][i]) + (part[q][2][i] + part[q][3][i]);
        d1[at] = a1[at] > 0.f ? r : 0.f;
    }
}

// Every parameter's gradient: gW[o][i] = sum_s dy[s][o] in(s, i), gb[o] = sum_s dy[s][o].
// A block takes 128 neighbouring parameters; the batch is split over WG_Q threads each.
constexpr int WG_P = 128, WG_Q = 8;
__global__ void __launch_bounds__(WG_P *WG_Q) k_mlp_wgrad(const float *__restrict__ X, const float *__restrict__ a1,
                                                         const float *__restrict__ a2, const float *__restrict__ d1,
                                                         const float *__restrict__ d2, const float *__restrict__ dout,
                                                         int B, float *__restrict__ grad) {
    __shared__ float part[WG_Q][WG_P];
    const int lp = threadIdx.x % WG_P, q = threadIdx.x / WG_P, p = blockIdx.x * WG_P + lp;
    float acc = 0.f;
    if (p < MLP_NPARAMS) {
        const float *dy, *x;
        int ldy, ldx, nin, r;  // r: the parameter within its layer's weights and biases
        bool relu = true;
        if (p < OFF_W2) {
            dy = d1, ldy = MLP_H, x = X, ldx = nin = MLP_IN, r = p, relu = false;
        } else if (p < OFF_W3) {
            dy = d2, ldy = MLP_H, x = a1, ldx = nin = MLP_H, r = p - OFF_W2;
        } else {
            dy = dout, ldy = MLP_OUT, x = a2, ldx = nin = MLP_H, r = p - OFF_W3;
        }
        const int nout = ldy;
        if (r < nout * nin) {
            dy += r / nin;
            x += r % nin;
#pragma unroll 8
            for (int s = q; s < B; s += WG_Q) {
                float v = x[(size_t)s * ldx];
                if (relu) v = fmaxf(v, 0.f);
                acc = fmaf(dy[(size_t)s * ldy], v, acc);
            }
        } else {
            dy += r - nout * nin;
#pragma unroll 8
            for (int s = q; s < B; s += WG_Q) acc += dy[(size_t)s * ldy];
        }
    }
    part[q][lp] = acc;
    __syncthreads();
    if (q == 0 && p < MLP_NPARAMS) {
        float r = part[0][lp];
#pragma unroll
        for (int k = 1; k < WG_Q; ++k) r += part[k][lp];
        grad[p] = r;
    }
}

__global__ void k_adam(float *theta, const float *g, float *m, float *v, int n, float lr, float c1, float c2) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float gi = g[i];
    const float mi = 0.9f * m[i] + 0.1f * gi;
    const float vi = 0.999f * v[i] + 0.001f * gi * gi;
    m[i] = mi;
    v[i] = vi;
    theta[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + 1e-8f);
}

// The 35 inputs from the moments of the scaled operator: Tr T_k / N for k < 32,
// emin/10, emax/10, N_e/N.
__global__ void k_features(const double *t, int64_t n_rows, double emin, double emax, double N_e, float *f) {
    const int i = threadIdx.x;
    if (i < 32) f[i] = (float)(t[i] / (double)n_rows);
    else if (i == 32) f[i] = (float)(emin / 10.0);
    else if (i == 33) f[i] = (float)(emax / 10.0);
    else if (i == 34) f[i] = (float)(N_e / (double)n_rows);
}

inline unsigned nb(int64_t n, int t = 128) { return (unsigned)((n + t - 1) / t); }

// Xavier-uniform initialisation: W ~ U(-a, a) with a = sqrt(6 / (fan_in +
// fan_out)) per layer, biases 0.  Uniforms from a counter-based generator:
// splitmix64 (Steele, Lea and Flood, "Fast splittable pseudorandom number
// generators", 2014) of (seed * 0xD1B54A32D192ED03) ^ i for parameter i, top 24
// bits + 1/2 scaled to (0, 1); the product a (2u - 1) is formed in FP64 and
// rounded once to FP32, so any IEEE host restatement gives the same bits.
__device__ __forceinline__ uint64_t mlp_splitmix64(uint64_t x) {
    uint64_t z = x + 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

__global__ void k_mlp_init(float *theta, uint64_t seed) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= MLP_NPARAMS) return;
    int fan = 0;  // fan_in + fan_out of the weight matrix holding i, 0 for a bias
    if (i < OFF_B1) fan = MLP_IN + MLP_H;
    else if (i >= OFF_W2 && i < OFF_B2) fan = MLP_H + MLP_H;
    else if (i >= OFF_W3 && i < OFF_B3) fan = MLP_H + MLP_OUT;
    if (fan == 0) {
        theta[i] = 0.f;
        return;
    }
    const uint64_t r = mlp_splitmix64((seed * 0xD1B54A32D192ED03ull) ^ (uint64_t)i);
    const double u = ((double)(r >> 40) + 0.5) * (1.0 / 16777216.0);
    const double lim = sqrt(6.0 / (double)fan);
    theta[i] = (float)(lim * (2.0 * u - 1.0));
}

}  // namespace cheb

using namespace cheb;

extern "C" int cheb_mlp_param_count(void) { return MLP_NPARAMS; }

extern "C" int cheb_mlp_init(float *theta, uint64_t seed, void *stream) {
    if (!theta) return fail(CHEB_ERR_INVALID, "cheb_mlp_init: theta is NULL");
    k_mlp_init<<<(MLP_NPARAMS + 255) / 256, 256, 0, as_stream(stream)>>>(theta, seed);
    return check_launch("k_mlp_init");
}

extern "C" int cheb_mlp_forward(const float *theta, const float *X, int32_t batch, float *act, float *out,
                                void *stream) {
    if (!theta || !X || !act || !out || batch < 1) return fail(CHEB_ERR_INVALID, "cheb_mlp_forward: bad arguments");
    cudaStream_t s = as_stream(stream);
    k_mlp_forward<<<nb(batch, MLP_S), MLP_NT, 0, s>>>(theta, X, batch, act, out);
    return check_launch("k_mlp_forward");
}

extern "C" int cheb_mlp_loss(const float *out, const float *xstar, const float *scale, int32_t batch, float *dout,
                             double *loss, void *stream) {
    if (!out || !xstar || !scale || !dout || batch < 1) return fail(CHEB_ERR_INVALID, "cheb_mlp_loss: bad arguments");
    k_mlp_loss<<<1, 256, 0, as_stream(stream)>>>(out, xstar, scale, batch, dout, loss);
    return check_launch("k_mlp_loss");
}

extern "C" int cheb_mlp_backward(const float *theta, const float *X, int32_t batch, const float *act,
                                 const float *dout, float *grad, float *ws, void *stream) {
    if (!theta || !X || !act || !dout || !grad || !ws || batch < 1)
        return fail(CHEB_ERR_INVALID, "cheb_mlp_backward: bad arguments");
    cudaStream_t s = as_stream(stream);
    const float *a1 = act, *a2 = act + (size_t)batch * MLP_H;
    float *d2 = ws, *d1 = ws + (size_t)batch * MLP_H;
    k_mlp_back<<<nb(batch, MLP_S), MLP_NT, 0, s>>>(theta, dout, a1, a2, batch, d1, d2);
    k_mlp_wgrad<<<nb(MLP_NPARAMS, WG_P), WG_P * WG_Q, 0, s>>>(X, a1, a2, d1, d2, dout, batch, grad);
    return check_launch("cheb_mlp_backward", 2);
}

extern "C" int cheb_mlp_adam(float *theta, const float *grad, float *m, float *v, int32_t t, float lr, void *stream) {
    if (!theta || !grad || !m || !v || t < 1) return fail(CHEB_ERR_INVALID, "cheb_mlp_adam: bad arguments");
    const float c1 = 1.f - powf(0.9f, (float)t), c2 = 1.f - powf(0.999f, (float)t);
    k_adam<<<nb(MLP_NPARAMS, 256), 256, 0, as_stream(stream)>>>(theta, grad, m, v, MLP_NPARAMS, lr, c1, c2);
    return check_launch("k_adam");
}

extern "C" int cheb_mlp_features(const double *moments, int64_t n_rows, double emin, double emax, double N_e,
                                 float *features, void *stream) {
    if (!moments || !features || n_rows < 1) return fail(CHEB_ERR_INVALID, "cheb_mlp_features: bad arguments");
    k_features<<<1, 64, 0, as_stream(stream)>>>(moments, n_rows, emin, emax, N_e, features);
    return check_launch("k_features");
}
