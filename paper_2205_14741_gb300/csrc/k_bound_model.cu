// Learned spectral bound: Lanczos labels and MLP training (the features and the
// inference run inside the gather kernel, k_pattern.cu).
//
// The network predicts, per submatrix A = T_j - mu I, the ratios rho/G and
// delta/G (spectral radius and smallest |eigenvalue| over the Gershgorin
// bound G) from nine cheap features; the Newton-Schulz start is then scaled
// with the predicted radius and checked against the guaranteed bound that the
// first product yields (see the Newton-Schulz kernels).  The paper's Section 4
// names learning on the fly (a network trained on data the simulation itself
// produces) as a direction; this is that reading for the sign iteration.
//
// Conventions shared with the FP64 oracle of the model (written separately):
//   features f0..f8 (all over G except f6 and f8):
//     ||A||_F/sqrt(n), max|A_rr|, mean|A_rr|, std(A_rr), max R_r, mean R_r,
//     n/256, mean A_rr, previous-step ratio;  R_r = sum_{c != r} |A_rc|
//   network F=9 -> 64 (tanh) -> 64 (tanh) -> 2, loss 1/(2m) sum (y - t)^2
//   flat parameters: W1 (64 x 9), b1, W2 (64 x 64), b2, W3 (2 x 64), b3
#include "smx_kernels.h"

namespace smx {

namespace {

constexpr int kF = kModelFeatures, kH = kModelHidden, kO = 2;

constexpr int kChunk = 64;  // samples per gradient block
constexpr int kGradThreads = 1024;  // kH units x kChunk / 4 samples
constexpr int kHs = kH + 1;  // row stride of W2 and h2 in shared memory: a column's entries lie in different banks

__device__ __forceinline__ float warp_sum_f(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

}  // namespace

// ---------------------------------------------------------------------------
// Lanczos labels (one CTA per submatrix): rho from A, delta from A^2
// ---------------------------------------------------------------------------
namespace {

// The i-th smallest eigenvalue (0-based) of the symmetric tridiagonal with diagonal a and off-diagonal
// b (b[0] unused), k <= kMaxLanczos, by one warp: each round counts the eigenvalues below 32 points of the
// current interval, a point per lane, and keeps the part that holds the i-th.  FP64 instructions take
// about 16 cycles per warp here however many lanes are active, so a round costs what one step of a
// bisection would and gains log2(33) bits instead of one: 11 rounds for 2^-55 of the starting interval.
// The count is the number of sign changes in the sequence of leading determinants p_j = (a_j - x) p_{j-1} -
// b_j^2 p_{j-2} (no division: three FP64 instructions a step), the matrix scaled by a power of two to
// norm 1 (entries a_j, -b_j^2 in `scaled`, the warp's own k of them) and the sequence rescaled before it
// can underflow.
__device__ double tridiag_eig(const double* a, const double* b, int k, int i, double2* scaled) {
    const int lane = threadIdx.x & 31;
    double lo = 1e300, hi = -1e300;
    for (int j = lane; j < k; j += 32) {
        const double r = (j ? fabs(b[j]) : 0.0) + (j + 1 < k ? fabs(b[j + 1]) : 0.0);
        lo = fmin(lo, a[j] - r);
        hi = fmax(hi, a[j] + r);
    }
    lo = -warp_max(-lo);
    hi = warp_max(hi);
    const int e = ilogb(fmax(fmax(fabs(lo), fabs(hi)), 1e-300)) + 1;
    const double sc = ldexp(1.0, -e);
    lo *= sc;
    hi *= sc;
    for (int j = lane; j < k; j += 32) {
        const double bj = j ? b[j] * sc : 0.0;
        scaled[j] = make_double2(a[j] * sc, -(bj * bj));
    }
    __syncwarp();
    for (int round = 0; round < 11 && hi > lo; ++round) {
        const double x = lo + (hi - lo) * (static_cast<double>(lane + 1) * (1.0 / 33.0));
        double p1 = 1.0, p0 = 0.0;  // p_{j-1}, p_{j-2}
        int cnt = 0;
        for (int j = 0; j < k; ++j) {
            const double2 ab = scaled[j];
            double p = fma(ab.x - x, p1, ab.y * p0);
            const int s1 = __double2hiint(p1) >> 31;
            // an exact zero counts as a sign change
            if (__double2loint(p) == 0 && (__double2hiint(p) & 0x7fffffff) == 0) p = s1 ? 1e-300 : -1e-300;
            cnt += (__double2hiint(p) >> 31) != s1;
            p0 = p1;
            p1 = p;
            if ((j & 3) == 3) {  // both small: up by 2^600 (an exponent added on the integer units)
                const int ex = max((__double2hiint(p0) >> 20) & 0x7ff, (__double2hiint(p1) >> 20) & 0x7ff);
                if (ex < 400) {
                    p0 *= 0x1p600;
                    p1 *= 0x1p600;
                }
            }
        }
        const unsigned above = __ballot_sync(0xffffffffu, cnt > i);  // the points right of the eigenvalue
        const int first = above ? __ffs(above) - 1 : 32;
        const double xl = __shfl_sync(0xffffffffu, x, first > 0 ? first - 1 : 0), xr = __shfl_sync(0xffffffffu, x, first & 31);
        if (first > 0) lo = xl;
        if (first < 32) hi = xr;
    }
    return ldexp(0.5 * (lo + hi), e);
}

}  // namespace

// STAGED: the submatrix is kept in shared memory (as FP32) for the up to 192 matrix-vector products
// that read it (144 at 48 steps): from L2 they took longer than anything but the eigenvalue searches.
// All 32 warps multiply (a row each, up to eight at a time); the vectors' sums stay with the first
// eight warps, whose order fixes their rounding.  Labels of 1024 submatrices (n 120 .. 204, 48
// steps) and 50 training steps: 23.3 ms from L2 with bisections by one thread, 6.3 ms staged and with
// multisection by a warp, 5.4 ms (3.9 of it here) with all warps on the products, 4.0 ms with the searches in
// k_lanczos_labels and eight warps in the vectors' barriers.
constexpr int kLanczosThreads = 1024, kLanczosVec = 256;
// a tridiagonal in global memory: diagonal, off-diagonal (entry 0 unused, one more at the end), size, and (the
// second one of a submatrix) the Gershgorin bound
constexpr int kTridiag = 2 * kMaxLanczos + 3;
static_assert(kTridiag == kLanczosTridiag, "doubles per tridiagonal");

template <class R, bool STAGED>
__global__ void __launch_bounds__(kLanczosThreads) k_lanczos(const SubDesc* __restrict__ subs, const R* __restrict__ T, int ksteps,
                                                             double* __restrict__ tridiag) {
    extern __shared__ float lz[];  // 4 vectors of n, then (STAGED) the submatrix
    __shared__ float red[8];
    __shared__ int last_s;
    __shared__ float gmax_s;
    const SubDesc s = subs[blockIdx.x];
    const R* t = T + s.t_off;
    const int n = s.n, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    float* v = lz;
    float* w = lz + n;
    float* vp = lz + 2 * n;
    float* u = lz + 3 * n;
    float* ts = lz + 4 * n;
    if constexpr (STAGED) {
        for (int r = warp; r < n; r += kLanczosThreads / 32)
#pragma unroll 4
            for (int c = lane; c < n; c += 32) ts[r * n + c] = static_cast<float>(t[static_cast<int64_t>(r) * s.ld + c]);
        __syncthreads();
    }
    auto entry = [&](int r, int c) -> float {
        if constexpr (STAGED) return ts[r * n + c];
        else return static_cast<float>(t[static_cast<int64_t>(r) * s.ld + c]);
    };

    // the sum of the first eight warps' values (called by them alone; a barrier of their own)
    auto vec_sync = [] { asm volatile("bar.sync 1, 256;" ::: "memory"); };
    auto block_sum_f = [&](float x) -> float {
        x = warp_sum_f(x);
        if (lane == 0) red[warp] = x;
        vec_sync();
        float r = 0.f;
        for (int i = 0; i < 8; ++i) r += red[i];
        vec_sync();
        return r;
    };
    // y = A x, kRows rows a warp at a time: each row's products summed over the lane's columns, then over the
    // lanes (the pairs of a butterfly, every pair added once: after three exchanges a lane holds one row)
    constexpr int kW = kLanczosThreads / 32, kRows = 8;
    auto matvec = [&](const float* x, float* y) {
        for (int r0 = warp; r0 < n; r0 += kW * kRows) {
            float acc[kRows];
            int row[kRows];  // (rows past n repeat row r0, not stored)
#pragma unroll
            for (int i = 0; i < kRows; ++i) {
                acc[i] = 0.f;
                row[i] = r0 + kW * i < n ? r0 + kW * i : r0;
            }
            for (int c = lane; c < n; c += 32) {
                const float xc = x[c];
#pragma unroll
                for (int i = 0; i < kRows; ++i)
                    if (i < 4 || r0 + kW * i < n) acc[i] = fmaf(entry(row[i], c), xc, acc[i]);  // (uniform over the warp)
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const bool up = lane & 16;
                const float send = up ? acc[i] : acc[i + 4], keep = up ? acc[i + 4] : acc[i];
                acc[i] = keep + __shfl_xor_sync(0xffffffffu, send, 16);
            }
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                const bool up = lane & 8;
                const float send = up ? acc[i] : acc[i + 2], keep = up ? acc[i + 2] : acc[i];
                acc[i] = keep + __shfl_xor_sync(0xffffffffu, send, 8);
            }
            const bool up = lane & 4;
            const float send = up ? acc[0] : acc[1], keep = up ? acc[1] : acc[0];
            float a = keep + __shfl_xor_sync(0xffffffffu, send, 4);
            a += __shfl_xor_sync(0xffffffffu, a, 2);
            a += __shfl_xor_sync(0xffffffffu, a, 1);
            const int mine = r0 + kW * (((lane & 16) ? 4 : 0) + ((lane & 8) ? 2 : 0) + ((lane & 4) ? 1 : 0));
            if ((lane & 3) == 0 && mine < n) y[mine] = a;
        }
        __syncthreads();
    };
    const bool vec = threadIdx.x < kLanczosVec;  // this thread works on the vectors' entries threadIdx.x, + 256, ...
    // Gershgorin bound G
    {
        float g = 0.f;
        for (int r = warp; r < n; r += kLanczosThreads / 32) {
            float acc = 0.f;
            for (int c = lane; c < n; c += 32) acc += fabsf(entry(r, c));
            g = fmaxf(g, warp_sum_f(acc));
        }
        if (threadIdx.x == 0) gmax_s = 0.f;
        __syncthreads();
        if (lane == 0) atomicMax(reinterpret_cast<int*>(&gmax_s), __float_as_int(g));  // (non-negative floats order like integers)
        __syncthreads();
    }
    const int K = min(ksteps, min(n, kMaxLanczos));
    double* tri = tridiag + static_cast<int64_t>(blockIdx.x) * 2 * kTridiag;  // A's tridiagonal, then A^2's
    for (int pass = 0; pass < 2; ++pass) {  // pass 0: A, pass 1: A^2
        // deterministic start vector with all components non-zero
        if (vec) {
            float nv = 0.f;
            for (int i = threadIdx.x; i < n; i += kLanczosVec) {
                v[i] = 1.0f + 0.5f * __sinf(1.7f * static_cast<float>(i) + 0.3f * pass);
                vp[i] = 0.f;
                nv += v[i] * v[i];
            }
            nv = sqrtf(block_sum_f(nv));
            for (int i = threadIdx.x; i < n; i += kLanczosVec) v[i] /= nv;
        }
        __syncthreads();
        float bprev = 0.f;
        int k = 0;
        for (; k < K; ++k) {
            if (pass == 0) matvec(v, w);
            else { matvec(v, u); matvec(u, w); }
            if (vec) {  // (an entry stays with its thread)
                float al = 0.f;
                for (int i = threadIdx.x; i < n; i += kLanczosVec) al += v[i] * w[i];
                al = block_sum_f(al);
                float nw = 0.f;
                for (int i = threadIdx.x; i < n; i += kLanczosVec) {
                    const float x = w[i] - al * v[i] - bprev * vp[i];
                    w[i] = x;
                    nw += x * x;
                }
                nw = sqrtf(block_sum_f(nw));
                const bool last = nw <= 1e-12f * gmax_s || k + 1 == K;
                if (threadIdx.x == 0) {
                    tri[k] = al;
                    tri[kMaxLanczos + k + 1] = nw;
                    last_s = last;
                }
                if (!last)
                    for (int i = threadIdx.x; i < n; i += kLanczosVec) {
                        vp[i] = v[i];
                        v[i] = w[i] / nw;
                    }
                bprev = nw;
            }
            __syncthreads();
            if (last_s) {
                ++k;
                break;
            }
        }
        if (threadIdx.x == 0) tri[2 * kMaxLanczos + 1] = k;
        tri += kTridiag;
        __syncthreads();
    }
    if (threadIdx.x == 0) tridiag[(static_cast<int64_t>(blockIdx.x) + 1) * 2 * kTridiag - 1] = gmax_s;
}

// The labels from the two tridiagonals of each submatrix: a warp finds the smallest and largest eigenvalue
// of A or the smallest of A^2 (three warps a submatrix, 3072 at a time in flight on 1024 submatrices:
// inside the Lanczos kernel, a CTA per SM, the latency of the FP64 recurrence was a third of its time).
__global__ void __launch_bounds__(96) k_lanczos_labels(const double* __restrict__ tridiag, float* __restrict__ labels) {
    __shared__ double2 scaled[3][kMaxLanczos];
    __shared__ double eig[3];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const double* tri = tridiag + static_cast<int64_t>(blockIdx.x) * 2 * kTridiag;
    const double* mine = tri + (warp == 2 ? kTridiag : 0);
    const int k = static_cast<int>(mine[2 * kMaxLanczos + 1]);
    const double x = tridiag_eig(mine, mine + kMaxLanczos, k, warp == 1 ? k - 1 : 0, scaled[warp]);
    if (lane == 0) eig[warp] = x;
    __syncthreads();
    if (threadIdx.x == 0) {
        const double g = tri[2 * kTridiag - 1], G = g > 0.0 ? g : 1.0;
        labels[2 * blockIdx.x] = static_cast<float>(fmax(fabs(eig[0]), fabs(eig[1])) / G);
        labels[2 * blockIdx.x + 1] = static_cast<float>(sqrt(fmax(eig[2], 0.0)) / G);
    }
}

// ---------------------------------------------------------------------------
// MLP
// ---------------------------------------------------------------------------

// Forward + backward for samples [blockIdx.x * 64, +64): per-block gradient sums
// (sum over the block's samples, in sample order) and half the squared residual.
// Bound by shared-memory reads; with rows of 64 words the lanes of a warp read W2 (a unit each) and h2 (a
// sample each) from one bank, 32 cycles a read.  So rows are 65 words apart, and a
// thread forms several outputs per read.  18.5 us for 1024 samples (16 CTAs: latency).
__global__ void __launch_bounds__(kGradThreads) k_mlp_grad(const float* __restrict__ params, const float* __restrict__ X,
                                                  const float* __restrict__ Tg, int m, float* __restrict__ partial,
                                                  float* __restrict__ partial_loss) {
    extern __shared__ __align__(16) float sm[];
    float* h1 = sm;                             // [64][64] (16-byte aligned, as d2)
    float* d2 = h1 + kChunk * kH;               // [64][64]
    float* d1 = d2 + kChunk * kH;               // [64][64]  dL/d(pre-activation 1)
    float* h2 = d1 + kChunk * kH;               // [64][65]
    float* w2 = h2 + kChunk * kHs;              // [64][65]  W2
    float* p = w2 + kH * kHs;                   // kModelParams
    float* xs = p + kModelParams;               // [64][kF]
    float* dy = xs + kChunk * kF;               // [64][2]
    float* ls = dy + kChunk * kO;               // [64] half squared residual per sample
    const int s0 = blockIdx.x * kChunk;
    const int cnt = min(kChunk, m - s0);
    for (int i = threadIdx.x; i < kModelParams; i += blockDim.x) {
        const float x = params[i];
        p[i] = x;
        if (i >= kOffW2 && i < kOffB2) w2[(i - kOffW2) / kH * kHs + (i - kOffW2) % kH] = x;
    }
    for (int i = threadIdx.x; i < kChunk * kF; i += blockDim.x) {
        const int sidx = i / kF;
        xs[i] = sidx < cnt ? X[static_cast<int64_t>(s0) * kF + i] : 0.f;
    }
    __syncthreads();
    // layer 1 and 2 forward: thread handles (sample, unit) pairs
    for (int e = threadIdx.x; e < kChunk * kH; e += blockDim.x) {
        const int sidx = e / kH, i = e - sidx * kH;
        float a = p[kOffB1 + i];
        for (int k = 0; k < kF; ++k) a = fmaf(p[i * kF + k], xs[sidx * kF + k], a);
        h1[e] = tanhf(a);
    }
    __syncthreads();
    // four samples a thread: a weight is read once for them, their h1 four units at a time
    const int unit = threadIdx.x & (kH - 1), four = 4 * (threadIdx.x / kH);
    {
        float a[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) a[u] = p[kOffB2 + unit];
#pragma unroll 4
        for (int k = 0; k < kH; k += 4) {
            float4 h[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) h[u] = *reinterpret_cast<const float4*>(h1 + (four + u) * kH + k);
            const float* wr = w2 + unit * kHs + k;
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                a[u] = fmaf(wr[0], h[u].x, a[u]);
                a[u] = fmaf(wr[1], h[u].y, a[u]);
                a[u] = fmaf(wr[2], h[u].z, a[u]);
                a[u] = fmaf(wr[3], h[u].w, a[u]);
            }
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) h2[(four + u) * kHs + unit] = tanhf(a[u]);
    }
    __syncthreads();
    if (threadIdx.x < kChunk * kO) {  // (a sample's outputs in neighbouring lanes)
        const int sidx = threadIdx.x >> 1, o = threadIdx.x & 1;
        float y = p[kOffB3 + o];
#pragma unroll 16
        for (int k = 0; k < kH; ++k) y = fmaf(p[kOffW3 + o * kH + k], h2[sidx * kHs + k], y);
        const float r = sidx < cnt ? y - Tg[2 * static_cast<int64_t>(s0 + sidx) + o] : 0.f;
        dy[sidx * kO + o] = r;
        const float r0 = __shfl_xor_sync(0xffffffffu, r, 1);
        if (o == 1) ls[sidx] = 0.5f * fmaf(r, r, r0 * r0);
    }
    __syncthreads();
    if (threadIdx.x == 0) {  // summed in sample order
        float l = 0.f;
#pragma unroll 16
        for (int i = 0; i < kChunk; ++i) l += ls[i];
        partial_loss[blockIdx.x] = l;
    }
    // backward: d2 = (dy W3) * (1 - h2^2); d1 = (d2 W2) * (1 - h1^2)
    for (int e = threadIdx.x; e < kChunk * kH; e += blockDim.x) {
        const int sidx = e / kH, i = e - sidx * kH;
        const float g = dy[sidx * kO] * p[kOffW3 + i] + dy[sidx * kO + 1] * p[kOffW3 + kH + i];
        const float h = h2[sidx * kHs + i];
        d2[e] = g * (1.f - h * h);
    }
    __syncthreads();
    {
        float g[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 4
        for (int i = 0; i < kH; i += 4) {
            float4 d[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) d[u] = *reinterpret_cast<const float4*>(d2 + (four + u) * kH + i);
            const float* wc = w2 + i * kHs + unit;
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                g[u] = fmaf(d[u].x, wc[0], g[u]);
                g[u] = fmaf(d[u].y, wc[kHs], g[u]);
                g[u] = fmaf(d[u].z, wc[2 * kHs], g[u]);
                g[u] = fmaf(d[u].w, wc[3 * kHs], g[u]);
            }
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int e = (four + u) * kH + unit;
            d1[e] = g[u] * (1.f - h1[e] * h1[e]);
        }
    }
    __syncthreads();
    // parameter gradients, each a sum over the block's samples in order
    float* gout = partial + static_cast<int64_t>(blockIdx.x) * kModelParams;
    {  // W2: rows four .. four + 3, column `unit`
        float g[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 4
        for (int sidx = 0; sidx < kChunk; ++sidx) {
            const float4 d = *reinterpret_cast<const float4*>(d2 + sidx * kH + four);
            const float h = h1[sidx * kH + unit];
            g[0] = fmaf(d.x, h, g[0]);
            g[1] = fmaf(d.y, h, g[1]);
            g[2] = fmaf(d.z, h, g[2]);
            g[3] = fmaf(d.w, h, g[3]);
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) gout[kOffW2 + (four + u) * kH + unit] = g[u];
    }
    for (int x = threadIdx.x; x < kModelParams - kH * kH; x += blockDim.x) {  // the others
        const int q = x < kOffW2 ? x : x + kH * kH;
        float g = 0.f;
        if (q < kOffB1) {
            const int i = q / kF, k = q - i * kF;
#pragma unroll 16
            for (int sidx = 0; sidx < kChunk; ++sidx) g = fmaf(d1[sidx * kH + i], xs[sidx * kF + k], g);
        } else if (q < kOffW2) {
            const int i = q - kOffB1;
            for (int sidx = 0; sidx < kChunk; ++sidx) g += d1[sidx * kH + i];
        } else if (q < kOffW3) {
            const int i = q - kOffB2;
            for (int sidx = 0; sidx < kChunk; ++sidx) g += d2[sidx * kH + i];
        } else if (q < kOffB3) {
            const int o = (q - kOffW3) / kH, k = (q - kOffW3) - o * kH;
            for (int sidx = 0; sidx < kChunk; ++sidx) g = fmaf(dy[sidx * kO + o], h2[sidx * kHs + k], g);
        } else {
            const int o = q - kOffB3;
            for (int sidx = 0; sidx < kChunk; ++sidx) g += dy[sidx * kO + o];
        }
        gout[q] = g;
    }
}

// Ordered sum of the block partials, divided by m; optional gradient output and
// optional Adam update (step t >= 1, lr > 0).
__global__ void k_mlp_reduce_adam(const float* __restrict__ partial, const float* __restrict__ partial_loss,
                                  int nblocks, int m, float* __restrict__ params, float* __restrict__ mst,
                                  float* __restrict__ vst, int t, float lr, float* __restrict__ grad_out,
                                  float* __restrict__ loss_out) {
    const int q = blockIdx.x * blockDim.x + threadIdx.x;
    const float inv_m = 1.f / static_cast<float>(m);
    if (q == 0 && loss_out) {
        float l = 0.f;
        for (int b = 0; b < nblocks; ++b) l += partial_loss[b];
        *loss_out = l * inv_m;
    }
    if (q >= kModelParams) return;
    float g = 0.f;
#pragma unroll 8
    for (int b = 0; b < nblocks; ++b) g += partial[static_cast<int64_t>(b) * kModelParams + q];
    g *= inv_m;
    if (grad_out) grad_out[q] = g;
    if (lr > 0.f) {
        const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
        const float mm = b1 * mst[q] + (1.f - b1) * g;
        const float vv = b2 * vst[q] + (1.f - b2) * g * g;
        mst[q] = mm;
        vst[q] = vv;
        const float mh = mm / (1.f - powf(b1, static_cast<float>(t)));
        const float vh = vv / (1.f - powf(b2, static_cast<float>(t)));
        params[q] -= lr * mh / (sqrtf(vh) + eps);
    }
}

// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------
template <class R>
static cudaError_t launch_lanczos_type(const SubDesc* subs, int n_subs, int max_n, const R* T, int ksteps, double* tridiag, float* labels,
                                       cudaStream_t st) {
    const size_t vectors = sizeof(float) * 4 * static_cast<size_t>(max_n), staged = vectors + sizeof(float) * static_cast<size_t>(max_n) * max_n;
    // up to n = 238 the submatrix fits shared memory
    const bool fits = staged <= 225u * 1024u;
    const size_t smem = fits ? staged : vectors;
    auto kernel = fits ? k_lanczos<R, true> : k_lanczos<R, false>;
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
    if (e != cudaSuccess) return e;
    kernel<<<n_subs, kLanczosThreads, smem, st>>>(subs, T, ksteps, tridiag);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    k_lanczos_labels<<<n_subs, 96, 0, st>>>(tridiag, labels);
    return cudaGetLastError();
}

cudaError_t launch_lanczos(const SubDesc* subs, int n_subs, int max_n, const void* T, bool fp32, int ksteps,
                           double* tridiag, float* labels, cudaStream_t st) {
    if (fp32) return launch_lanczos_type(subs, n_subs, max_n, static_cast<const float*>(T), ksteps, tridiag, labels, st);
    return launch_lanczos_type(subs, n_subs, max_n, static_cast<const double*>(T), ksteps, tridiag, labels, st);
}

size_t mlp_partial_floats(int m) { return static_cast<size_t>((m + kChunk - 1) / kChunk) * (kModelParams + 1); }

cudaError_t launch_mlp_step(const float* params_in, const float* X, const float* Tg, int m, float* partial,
                            float* params, float* mst, float* vst, int t, float lr, float* grad_out, float* loss_out,
                            cudaStream_t st) {
    if (m <= 0) return cudaErrorInvalidValue;
    const int nb = (m + kChunk - 1) / kChunk;
    float* partial_loss = partial + static_cast<size_t>(nb) * kModelParams;
    const size_t smem = sizeof(float) * (kModelParams + kChunk * kF + 3 * kChunk * kH + kChunk * kHs + kH * kHs + kChunk * kO + kChunk);
    cudaError_t e = cudaFuncSetAttribute(k_mlp_grad, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
    if (e != cudaSuccess) return e;
    k_mlp_grad<<<nb, kGradThreads, smem, st>>>(params_in, X, Tg, m, partial, partial_loss);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    k_mlp_reduce_adam<<<(kModelParams + 255) / 256, 256, 0, st>>>(partial, partial_loss, nb, m, params, mst, vst, t, lr,
                                                                  grad_out, loss_out);
    return cudaGetLastError();
}

}  // namespace smx
