// The 64-bit forms in FP64 arithmetic, for submatrices whose rows are of very different size.
//
// Floating point keeps the relative precision of small rows through a product; the fixed point of the digit slices
// (smx_slices.cuh) holds every entry in units of the submatrix's largest row.  For A = D S0 D with a well-conditioned
// S0 the relative error of A^-1/2 stays at some 1e-15 in the one and grows as 1 / d^2 in the other (d the smallest
// entry of D).  So the kernels of k_ns_fp64.cu put such submatrices on a list (kGraded there says which) and leave
// them to the kernels below, which follow every launch of those and return at once when the list is empty (a build's
// also forms the sums of its partials, which had a launch of their own; dense n = 192 275 -> 277 us).
//
// A persistent CTA takes one submatrix at a time and keeps its matrices in a slot of the other kernels' work memory.
// Bound by the FP64 units, which take about 16 cycles per warp instruction and SM: products in 64 x 64 tiles from
// shared memory, 2 x 4 entries per thread, with no work for the padding beyond 4 rows and 16 columns.  A density build
// of 256 submatrices (n = 161 on average, 21 steps): 137 ms (231 ms with work for the padding to 64); by the slices
// the steps of as many submatrices take a twenty-fourth of the time.
#include "smx_finish.cuh"
#include "smx_kernels.h"

namespace smx {

namespace {

constexpr int kThreads = 512, kWarps = kThreads / 32;
constexpr int kTile = 64, kKc = 16;

// The work matrices of one submatrix (n x n, leading dimension n) and the CTA's shared memory.
struct Work {
    int n;
    double* buf[5];
    double (*As)[kTile + 1];
    double (*Bs)[kTile + 1];
    double* scratch;  // 64 doubles

};

template <class F>
__device__ __forceinline__ void each(int n, F f) {  // f(r, c) for every entry, a warp to a row
    for (int r = threadIdx.x >> 5; r < n; r += kWarps)
        for (int c = threadIdx.x & 31; c < n; c += 32) f(r, c);
    __syncthreads();
}

// C = dg I + cf A B (n x n row by row, leading dimensions lda, ldb and ldc).  Returns this thread's share of
// ||A B - I||_F^2.
__device__ __noinline__ double product(const Work& w, const double* A, int lda, const double* B, int ldb, double* C, int ldc, double cf, double dg) {
    const int n = w.n, tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    double r2 = 0.0;
    for (int r0 = 0; r0 < n; r0 += kTile)
        for (int c0 = 0; c0 < n; c0 += kTile) {
            const bool rows = r0 + 4 * (tid >> 5) < n;  // the warp's four rows
            double acc[2][4] = {};
            for (int k0 = 0; k0 < n; k0 += kKc) {
                for (int e = tid; e < kTile * kKc; e += kThreads) {
                    const int rr = e / kKc, kk = e % kKc;
                    w.As[kk][rr] = r0 + rr < n && k0 + kk < n ? A[static_cast<int64_t>(r0 + rr) * lda + k0 + kk] : 0.0;
                }
                for (int e = tid; e < kTile * kKc; e += kThreads) {
                    const int kk = e / kTile, cc = e % kTile;
                    w.Bs[kk][cc] = k0 + kk < n && c0 + cc < n ? B[static_cast<int64_t>(k0 + kk) * ldb + c0 + cc] : 0.0;
                }
                __syncthreads();
                if (rows)
#pragma unroll
                    for (int kk = 0; kk < kKc; ++kk) {
                        const double a0 = w.As[kk][2 * ty], a1 = w.As[kk][2 * ty + 1];
#pragma unroll
                        for (int j = 0; j < 4; ++j)
                            if (c0 + 16 * j < n) {
                                const double b = w.Bs[kk][tx + 16 * j];
                                acc[0][j] = fma(a0, b, acc[0][j]);
                                acc[1][j] = fma(a1, b, acc[1][j]);
                            }
                    }
                __syncthreads();
            }
#pragma unroll
            for (int i = 0; i < 2; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const int row = r0 + 2 * ty + i, col = c0 + tx + 16 * j;
                    if (row >= n || col >= n) continue;
                    const double v = acc[i][j], one = row == col ? 1.0 : 0.0;
                    C[static_cast<int64_t>(row) * ldc + col] = dg * one + cf * v;
                    r2 += (v - one) * (v - one);
                }
        }
    __syncthreads();
    return r2;
}
__device__ __forceinline__ double product(const Work& w, const double* A, const double* B, double* C, double cf, double dg) {
    return product(w, A, w.n, B, w.n, C, w.n, cf, dg);
}

// C[i m + q] = scale (A B)[i][q] for i < n, q < m, with B[k][q] = Bt[q sq + k sk]; rest: scale (B - A B) instead.
// A warp per row i, eight columns at a time.
__device__ __noinline__ void thin_product(int n, const double* A, int lda, const double* Bt, int64_t sq, int64_t sk, int m, double* C, bool rest,
                                          double scale) {
    const int lane = threadIdx.x & 31;
    for (int i = threadIdx.x >> 5; i < n; i += kWarps)
        for (int q0 = 0; q0 < m; q0 += 8) {
            double acc[8] = {};
            for (int k = lane; k < n; k += 32) {
                const double x = A[static_cast<int64_t>(i) * lda + k];
#pragma unroll
                for (int t = 0; t < 8; ++t)
                    if (q0 + t < m) acc[t] = fma(x, Bt[(q0 + t) * sq + k * sk], acc[t]);
            }
#pragma unroll
            for (int t = 0; t < 8; ++t) {
                const double v = warp_sum(acc[t]);
                if (lane == 0 && q0 + t < m) C[static_cast<int64_t>(i) * m + q0 + t] = scale * (rest ? Bt[(q0 + t) * sq + i * sk] - v : v);
            }
        }
    __syncthreads();
}

struct SignResult {
    double *X, *Z, *Y;  // the last iterate; the others are free
    double rmax, scale;  // the largest row sum of |X0^2| and the factor of the first step
    int done;
    bool conv, bad;
};

// Newton-Schulz steps X <- X (3/2 I - 1/2 X^2) from X0 = (src - mu I) / b; the scaling after the first product and the
// learned bound's rules are those of sign_steps (dhat: the predicted smallest |eigenvalue| of X0, negative: none).
__device__ SignResult sign_iteration(const Work& w, const double* src, int ld, double mu, double b, bool use_model, double dhat, int* fallbacks,
                                     int max_iter, double tau) {
    const int n = w.n, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    SignResult s{w.buf[0], w.buf[2], w.buf[1], 0.0, 1.0, 0, false, false};
    double* const Y = s.Y;
    const double inv_b = 1.0 / b;
    each(n, [&](int r, int c) { s.X[static_cast<int64_t>(r) * n + c] = (src[static_cast<int64_t>(r) * ld + c] - (r == c ? mu : 0.0)) * inv_b; });
    double lsch = 1.0;
    for (int it = 0; it < max_iter; ++it) {
        double r2 = 1.0, oscale = 1.0, acur = 1.0;
        if (it == 0) {
            product(w, s.X, s.X, Y, 1.0, 0.0);
            // rho(X0)^2 <= max_r (|Y| v)_r / v_r for v = 1 and two power steps from it (v in the second product's buffer
            // and the one after it)
            double *v = s.Z, *next = w.buf[3];
            auto max2 = [&](double x, double y) -> double2 {
                x = warp_max(x);
                y = warp_max(y);
                if (lane == 0) {
                    w.scratch[warp] = x;
                    w.scratch[32 + warp] = y;
                }
                __syncthreads();
                double2 m = make_double2(0.0, 0.0);
                for (int i = 0; i < kWarps; ++i) {
                    m.x = fmax(m.x, w.scratch[i]);
                    m.y = fmax(m.y, w.scratch[32 + i]);
                }
                __syncthreads();
                return m;
            };
            double rmax = 0.0;
            for (int r = warp; r < n; r += kWarps) {
                double acc = 0.0;
                for (int c = lane; c < n; c += 32) acc += fabs(Y[static_cast<int64_t>(r) * n + c]);
                acc = warp_sum(acc);
                if (lane == 0) v[r] = acc;
                rmax = fmax(rmax, acc);
            }
            rmax = max2(rmax, 0.0).x;
            double best = rmax, top = rmax;
            for (int pass = 0; pass < 2 && best > 0.0; ++pass) {
                for (int c = threadIdx.x; c < n; c += kThreads) v[c] = fmax(v[c], 1e-30 * top);
                __syncthreads();
                double q = 0.0, most = 0.0;
                for (int r = warp; r < n; r += kWarps) {
                    double acc = 0.0;
                    for (int c = lane; c < n; c += 32) acc = fma(fabs(Y[static_cast<int64_t>(r) * n + c]), v[c], acc);
                    acc = warp_sum(acc);
                    if (lane == 0) next[r] = acc;
                    q = fmax(q, acc / v[r]);
                    most = fmax(most, acc);
                }
                const double2 m2 = max2(q, most);
                best = fmin(best, m2.x);
                if (!(m2.y > 0.0)) break;
                for (int c = threadIdx.x; c < n; c += kThreads) v[c] = next[c] / m2.y;
                top = 1.0;
            }
            const double smax = sqrt(best * (1.0 + 1e-12));
            double scale = smax > 0.0 ? 1.2 / smax : 1.0;
            if (use_model && smax > 0.0) {
                const bool gap = dhat > 0.0;
                if (gap ? dhat <= smax : smax <= 1.7) {
                    if (gap) {  // the scaled schedule from l0 = dhat / s
                        const double l0 = dhat / smax, a0 = ns_scale(l0);
                        scale = a0 / smax;
                        lsch = ns_next_lower(a0, l0);
                    } else {
                        scale = fmax(1.0, scale);
                    }
                } else if (threadIdx.x == 0) {
                    atomicAdd(fallbacks, 1);
                }
            }
            s.rmax = rmax;
            s.scale = oscale = scale;
            each(n, [&](int r, int c) {
                double& y = Y[static_cast<int64_t>(r) * n + c];
                y = (r == c ? 1.5 : 0.0) - 0.5 * scale * scale * y;
            });
        } else {
            // Y = a (3/2 I - a^2/2 X^2) on the scaled schedule (a = 1: a plain step)
            double cf = -0.5, dg = 1.5;
            if (lsch < 1.0) {
                const double f = ns_scale(lsch);
                cf = -0.5 * f * f * f;
                dg = 1.5 * f;
                lsch = ns_next_lower(f, lsch);
                acur = f;
            }
            r2 = block_sum(product(w, s.X, s.X, Y, cf, dg), w.scratch);
        }
        product(w, s.X, Y, s.Z, oscale, 0.0);
        double* t = s.X;
        s.X = s.Z;
        s.Z = t;
        s.done = it + 1;
        if (!isfinite(r2)) {
            s.bad = true;
            break;
        }
        if (it > 0 && sqrt(r2) <= tau) {
            // stop after this step unless it was a scaled step whose factor moves converged eigenvalues off 1
            if (acur - 1.0 <= 2e-6) {
                s.conv = true;
                break;
            }
            lsch = 1.0;
        }
    }
    return s;
}

struct RootResult {
    double *Y, *Z, *T;  // (A / b)^1/2, (A / b)^-1/2 and a free buffer
    int done;
    bool conv, bad;
};

// The coupled iteration: T = 3/2 I - 1/2 Z Y, Y <- Y T, Z <- T Z from Y = src / b and Z = I.  What is not positive
// definite overflows.
__device__ RootResult root_iteration(const Work& w, const double* src, int ld, double b, int max_iter, double tau) {
    const int n = w.n;
    RootResult s{w.buf[0], w.buf[1], w.buf[2], 0, false, false};
    double* N = w.buf[3];
    const double inv_b = 1.0 / b;
    each(n, [&](int r, int c) {
        s.Y[static_cast<int64_t>(r) * n + c] = src[static_cast<int64_t>(r) * ld + c] * inv_b;
        s.Z[static_cast<int64_t>(r) * n + c] = r == c ? 1.0 : 0.0;
    });
    for (int it = 0; it < max_iter; ++it) {
        const double r2 = block_sum(product(w, s.Z, s.Y, s.T, -0.5, 1.5), w.scratch);
        product(w, s.Y, s.T, N, 1.0, 0.0);    // Y'
        product(w, s.T, s.Z, s.Y, 1.0, 0.0);  // Z' into Y's buffer
        double* old = s.Z;
        s.Z = s.Y;
        s.Y = N;
        N = old;
        s.done = it + 1;
        if (!isfinite(r2)) {
            s.bad = true;
            break;
        }
        if (it > 0 && sqrt(r2) <= tau) {
            s.conv = true;
            break;
        }
    }
    return s;
}

// The Fermi function's T = tanh(beta A / 2) (fermi_tanh in k_ns_fp64.cu) for g >= the spectral radius of A: the Taylor
// start and k doublings tanh(2x) = 2 tanh(x) / (1 + tanh(x)^2), the inverse of M = I + T^2 by Newton-Schulz V <- V +
// V (I - M V) from V = 4/3 I - 4/9 M until ||I - M V||_F <= 1e-15 sqrt(n).  Returns T's buffer, counts the products.
__device__ double* tanh_doublings(const Work& w, const double* src, int ld, double g, double beta, int& products, bool& bad) {
    const int n = w.n;
    bad = false;
    products = 0;
    int k = 0;
    double sc = 0.5 * beta * g;
    while (sc > 1.0 / 16.0 && k < 60) {
        sc *= 0.5;
        ++k;
    }
    auto at = [&](int r, int c) -> int64_t { return static_cast<int64_t>(r) * n + c; };
    auto prod = [&](const double* A, const double* B, double* C, double cf, double dg) {
        ++products;
        return product(w, A, B, C, cf, dg);
    };
    double *X = w.buf[0], *Y = w.buf[1], *P = w.buf[2], *T = w.buf[3];
    const double f = sc / g;
    each(n, [&](int r, int c) { X[at(r, c)] = src[static_cast<int64_t>(r) * ld + c] * f; });
    prod(X, X, Y, 1.0, 0.0);
    const double cs[6] = {1.0, -1.0 / 3.0, 2.0 / 15.0, -17.0 / 315.0, 62.0 / 2835.0, -1382.0 / 155925.0};
    each(n, [&](int r, int c) { P[at(r, c)] = cs[5] * Y[at(r, c)] + (r == c ? cs[4] : 0.0); });
    for (int i = 3; i >= 0; --i) {
        prod(P, Y, T, 1.0, cs[i]);
        double* t = P;
        P = T;
        T = t;
    }
    prod(X, P, T, 1.0, 0.0);
    double* fr[4] = {X, Y, P, w.buf[4]};  // free buffers
    for (int d = 0; d < k && !bad; ++d) {
        double *M = fr[0], *V = fr[1], *R = fr[2], *W = fr[3];
        prod(T, T, M, 1.0, 1.0);  // I + T^2
        each(n, [&](int r, int c) { V[at(r, c)] = (r == c ? 4.0 / 3.0 : 0.0) - 4.0 / 9.0 * M[at(r, c)]; });
        for (int m = 0; m < 12; ++m) {
            const double r2 = block_sum(prod(M, V, R, -1.0, 1.0), w.scratch);  // R = I - M V
            if (!isfinite(r2)) {
                bad = true;
                break;
            }
            if (sqrt(r2) <= 1e-15 * sqrt(static_cast<double>(n))) break;
            prod(V, R, W, 1.0, 0.0);
            each(n, [&](int r, int c) { W[at(r, c)] += V[at(r, c)]; });  // V + V R
            double* t = V;
            V = W;
            W = t;
        }
        prod(T, V, R, 2.0, 0.0);
        fr[0] = T;
        fr[1] = M;
        fr[2] = V;
        fr[3] = W;
        T = R;
    }
    return T;
}

// The next listed submatrix (its place in the list, every thread gets it).
__device__ __forceinline__ int next_listed(GradedList* list, int* job_s) {
    __syncthreads();
    if (threadIdx.x == 0) *job_s = atomicAdd(&list->next, 1);
    __syncthreads();
    return *job_s;
}
// The last CTA empties the list, and gets true (job_s: a word of shared memory).
__device__ __forceinline__ bool release_list(GradedList* list, int* job_s) {
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
        *job_s = atomicAdd(&list->done, 1) == static_cast<int>(gridDim.x) - 1;
        if (*job_s) list->count = list->next = list->done = 0;
    }
    __syncthreads();
    __threadfence();
    return *job_s != 0;
}

__device__ __forceinline__ Work slot_work(int n, uint8_t* slot, double (*As)[kTile + 1], double (*Bs)[kTile + 1], double* scratch) {
    Work w;
    w.n = n;
    for (int i = 0; i < 5; ++i) w.buf[i] = reinterpret_cast<double*>(slot + kSlotHead) + static_cast<int64_t>(i) * n * n;
    w.As = As;
    w.Bs = Bs;
    w.scratch = scratch;
    return w;
}

}  // namespace

// The listed submatrices of a build, then (the last CTA; the first if none is listed) the sums of its partials.
__global__ void __launch_bounds__(kThreads) k_ns_graded(const __grid_constant__ NsFp64Args a) {
    __shared__ double As[kKc][kTile + 1], Bs[kKc][kTile + 1], scratch[64];
    __shared__ SubDesc s;
    __shared__ int job_s;
    extern __shared__ int ls_smem[];
    if (a.skip && *a.skip) return;
    const int count = a.graded->count;
    if (count == 0) {
        if (a.sums && blockIdx.x == 0) sum_partials(a.partial, a.n_cols, &a.sums->trace, &a.sums->energy, scratch);
        return;
    }
    uint8_t* slot = a.ws + static_cast<int64_t>(blockIdx.x) * a.slot_bytes;
    for (;;) {
        const int job = next_listed(a.graded, &job_s);
        if (job >= count) break;
        if (threadIdx.x == 0) s = a.subs[a.graded->column[job]];
        __syncthreads();
        const int j = s.col, n = s.n;
        const Work w = slot_work(n, slot, As, Bs, scratch);
        const double* T = a.T + s.t_off;
        const int64_t own = static_cast<int64_t>(s.own) * n;
        auto record = [&](int done, bool conv, bool bad) {
            if (threadIdx.x != 0) return;
            a.iters[j] = done;
            atomicAdd(a.work_n3, static_cast<unsigned long long>(n) * n * n * done);
            if (bad) atomicCAS(a.status, kOk, kErrNonfinite);
            else if (!conv) atomicCAS(a.status, kOk, kErrNoconv);
        };
        if (a.function == kFnFermi) {
            int products;
            bool bad;
            const double* F = tanh_doublings(w, T, s.ld, a.bound[j], a.beta, products, bad);
            record(products, true, bad);
            auto row = [&](int q, int i) -> double { return bad ? NAN : F[own + static_cast<int64_t>(q) * n + i]; };
            finish_column(s, a.pv, a.H, a.D, a.partial, row, ls_smem, scratch);  // 1/2 (I - T)
        } else if (a.function != kFnDensity) {
            // A^-1/2 = Z / sqrt(b), A^1/2 = sqrt(b) Y, A^-1 = Z Z / b
            const double b = a.bound[j];
            const RootResult r = root_iteration(w, T, s.ld, b, a.max_iter, a.tau);
            record(r.done, r.conv, r.bad);
            const bool inv = a.function == kFnInv;
            if (inv) thin_product(n, r.Z, n, r.Z + own, n, 1, s.bown, r.T, false, 1.0 / b);
            const double* F = inv ? r.T : (a.function == kFnSqrt ? r.Y : r.Z) + own;
            const double fs = r.bad ? NAN : inv ? 1.0 : a.function == kFnSqrt ? sqrt(b) : 1.0 / sqrt(b);
            const int64_t sq = inv ? 1 : n, si = inv ? s.bown : 1;
            auto row = [&](int q, int i) -> double { return fs * F[q * sq + i * si]; };
            finish_column(s, a.pv, a.H, a.D, a.partial, row, ls_smem, scratch, false);
        } else {
            const double gersh = a.gersh[j], b = a.Mc ? gersh : a.bound[j];
            const SignResult r = sign_iteration(w, (a.Mc ? a.Mc : a.T) + s.t_off, s.ld, a.Mc ? a.mu : 0.0, b, a.use_model != 0,
                                                a.pred ? static_cast<double>(a.pred[2 * j + 1]) * gersh / b : -1.0, a.fallbacks, a.max_iter, a.tau);
            record(r.done, r.conv, r.bad);
            if (threadIdx.x == 0) {
                a.sq_ratio[j] = static_cast<float>(sqrt(r.rmax) * b / gersh);
                a.bound[j] = b / r.scale;
            }
            if (a.Mc) {  // 1/2 L (W - X W), W = L[:, own] (rows own .. of the symmetric L)
                const double* L = a.Lc + s.t_off;
                thin_product(n, r.X, n, L + static_cast<int64_t>(s.own) * s.ld, s.ld, 1, s.bown, r.Y, true, 1.0);
                thin_product(n, L, s.ld, r.Y, 1, s.bown, s.bown, r.Z, false, 0.5);
                auto row = [&](int q, int i) -> double { return r.bad ? NAN : r.Z[static_cast<int64_t>(i) * s.bown + q]; };
                finish_column(s, a.pv, a.H, a.D, a.partial, row, ls_smem, scratch, false, a.Sv);
            } else {
                auto row = [&](int q, int i) -> double { return r.bad ? NAN : r.X[own + static_cast<int64_t>(q) * n + i]; };
                finish_column(s, a.pv, a.H, a.D, a.partial, row, ls_smem, scratch);
            }
        }
    }
    if (release_list(a.graded, &job_s) && a.sums) sum_partials(a.partial, a.n_cols, &a.sums->trace, &a.sums->energy, scratch);
}

// The listed submatrices of a non-orthogonal setup: L = A_S^-1/2 into Lc, M = L A_H L into Mc and its interval.
__global__ void __launch_bounds__(kThreads) k_graded_setup(const __grid_constant__ NonorthSetupArgs a) {
    __shared__ double As[kKc][kTile + 1], Bs[kKc][kTile + 1], scratch[64];
    __shared__ SubDesc s;
    __shared__ int job_s;
    const int count = a.graded->count;
    if (count == 0) return;
    uint8_t* slot = a.ws + static_cast<int64_t>(blockIdx.x) * a.slot_bytes;
    for (;;) {
        const int job = next_listed(a.graded, &job_s);
        if (job >= count) break;
        if (threadIdx.x == 0) s = a.subs[a.graded->column[job]];
        __syncthreads();
        const int n = s.n, ld = s.ld;
        const Work w = slot_work(n, slot, As, Bs, scratch);
        double *Lc = a.Lc + s.t_off, *Mc = a.Mc + s.t_off;
        const double b = a.bound_s[s.col];
        const RootResult r = root_iteration(w, Lc, ld, b, a.max_iter, a.tau);
        if (threadIdx.x == 0) {
            a.iters[s.col] = r.done;
            a.root_graded[s.col] = 1;
            if (r.bad) atomicCAS(a.status, kOk, kErrNonfinite);
            else if (!r.conv) atomicCAS(a.status, kOk, kErrNoconv);
        }
        const double ls = 1.0 / sqrt(b);
        each(n, [&](int i, int c) { Lc[static_cast<int64_t>(i) * ld + c] = ls * r.Z[static_cast<int64_t>(i) * n + c]; });
        product(w, Mc, ld, Lc, ld, r.T, n, 1.0, 0.0);   // A_H L
        product(w, Lc, ld, r.T, n, r.Y, n, 1.0, 0.0);   // L A_H L
        each(n, [&](int i, int c) {
            Mc[static_cast<int64_t>(i) * ld + c] = 0.5 * (r.Y[static_cast<int64_t>(i) * n + c] + r.Y[static_cast<int64_t>(c) * n + i]);
        });
        // its Gershgorin interval
        const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
        double lo = INFINITY, hi = -INFINITY;
        for (int i = warp; i < n; i += kWarps) {
            double acc = 0.0;
            for (int c = lane; c < n; c += 32) acc += c == i ? 0.0 : fabs(Mc[static_cast<int64_t>(i) * ld + c]);
            acc = warp_sum(acc);
            const double d = Mc[static_cast<int64_t>(i) * ld + i];
            lo = fmin(lo, d - acc);
            hi = fmax(hi, d + acc);
        }
        if (lane == 0) {
            scratch[warp] = lo;
            scratch[32 + warp] = hi;
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            for (int i = 1; i < kWarps; ++i) {
                lo = fmin(lo, scratch[i]);
                hi = fmax(hi, scratch[32 + i]);
            }
            a.lohi[2 * s.col] = r.bad ? 0.0 : lo;
            a.lohi[2 * s.col + 1] = r.bad ? 0.0 : hi;
        }
    }
    release_list(a.graded, &job_s);
}

// The dense entry point's matrix, when *graded (cleared here) says that its rows are of very different size: D = 1/2 (I
// - sign(H - mu I)) with rows of H - mu I of at most b; status gets the result, work holds three n x n matrices and a row.
__global__ void __launch_bounds__(kThreads) k_dense_graded(const double* __restrict__ H, int n, double mu, double* __restrict__ D, uint8_t* slot,
                                                           double tau, int max_iter, int* graded, const double* b, int* status) {
    __shared__ double As[kKc][kTile + 1], Bs[kKc][kTile + 1], scratch[64];
    if (*graded == 0) return;
    const Work w = slot_work(n, slot, As, Bs, scratch);
    const SignResult r = sign_iteration(w, H, n, mu, *b, false, -1.0, nullptr, max_iter, tau);
    each(n, [&](int i, int c) {
        D[static_cast<int64_t>(i) * n + c] = r.bad ? NAN : 0.5 * ((i == c ? 1.0 : 0.0) - r.X[static_cast<int64_t>(i) * n + c]);
    });
    if (threadIdx.x == 0) {
        status[0] = r.bad ? kErrNonfinite : r.conv ? kOk : kErrNoconv;
        status[1] = r.done;
    }
}

cudaError_t launch_ns_graded(const NsFp64Args& a, int slots, int max_nblk, cudaStream_t st) {
    const size_t smem = sizeof(int) * (static_cast<size_t>(max_nblk) + 1);
    if (smem > (16u << 10)) {  // (beside 17 KB of static arrays)
        const cudaError_t e = cudaFuncSetAttribute(k_ns_graded, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
        if (e != cudaSuccess) return e;
    }
    k_ns_graded<<<slots, kThreads, smem, st>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_graded_setup(const NonorthSetupArgs& a, int slots, cudaStream_t st) {
    k_graded_setup<<<slots, kThreads, 0, st>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_dense_graded(const double* H, int n, double mu, double* D, uint8_t* slot, double tau, int max_iter, int* graded, const double* b,
                                int* status, cudaStream_t st) {
    cudaLaunchConfig_t cfg = {};  // (an error of the caller's that is pending is neither taken for one of this launch nor cleared)
    cfg.gridDim = dim3(1);
    cfg.blockDim = dim3(kThreads);
    cfg.stream = st;
    return cudaLaunchKernelEx(&cfg, k_dense_graded, H, n, mu, D, slot, tau, max_iter, graded, b, status);
}

}  // namespace smx
