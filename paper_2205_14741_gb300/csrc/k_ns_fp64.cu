// Newton-Schulz sign iteration in 64-bit arithmetic (the plain form), and the function forms.
//
// Eq. 13 defines sign(A) = A (A^2)^(-1/2).  The iteration
//     X_{k+1} = 1/2 X_k (3 I - X_k^2) = X_k + 1/2 X_k W_k,   W_k = I - X_k^2,
// converges to sign(T_j - mu I) when every eigenvalue of X_0 (a multiple of T_j - mu I) lies in
// (-sqrt 3, 0) u (0, sqrt 3).  Each step is two symmetric products; the first also yields the
// residual ||X^2 - I||_F.  Stopping rule: after the step whose residual is <= tau (the next
// residual is ~0.75 tau^2).
//
// The products run on the tensor cores by error-free slices (smx_slices.cuh), and everything
// between them is 64-bit integer arithmetic in units of 2^-62: GB300's FP64 units take about 16
// cycles per warp instruction, so one FP64 operation per matrix entry costs as much as a quarter of
// a product (n = 158).  One persistent CTA per SM (or cluster of CTAs, where there are fewer
// submatrices than SMs: launch_form) takes submatrices largest first and keeps an iterate, one product
// and the operands' digits in a slot of global memory (152 slots of 1.1 MB in use at k = 160: about
// half of the accesses hit L2, DRAM runs at 43 %).
//
// Measured with products on the FP64 units (64 x 64 tiles, 4 x 4 per thread) and this way: a density build of
// 1024 submatrices (n 120 .. 204) 164 and 6.5 ms, the inverse square root 206 and 7.5 ms, the Fermi function of 128
// (n 138 .. 240) 528 and 16.4 ms.  Of a submatrix's time 60 % are products, 27 % the passes between them (bound by
// issue: some 500 instructions for eight entries), the rest loading and the bound.
#include <climits>

#include "smx_finish.cuh"
#include "smx_kernels.h"
#include "smx_slices.cuh"

namespace smx {

namespace {

// The matrices of one submatrix in its CTA's slot: k x k integers (units of 2^-62) and digit planes.
struct SliceJob {
    int n, k;  // dimension, and rounded up to 32 (rows and columns past n are zero)
    int64_t* M[kFp64Mats];
    uint8_t* P[kFp64Planes];
    float* scratch;  // of the cluster (the first kSlotHead bytes of its slot): sums, maxima, the claimed job, maxima
    unsigned long long* sums;  // of the cluster: three squared lengths per row (coupled_steps)
};

// Scalars that one thread forms in FP64 for the CTA.
struct SliceScalars {
    int job;
    int e;
    int bad;
    int graded;        // the rows of the matrix looked at last are of very different size (kGraded)
    int stop;          // the schedule's factor allows this step to be the last
    uint64_t f1, f2;   // the step's factor a and a^2 (fixed_factor), 0 for a plain step
    double lsch;       // lower end of the interval the scaled schedule assumes (1: plain steps)
    unsigned long long u[kSliceWarps];
    double d[kSliceWarps];
};

__device__ __forceinline__ void slice_job(SliceJob& jb, uint8_t* slot, int n, int kmax, int mats) {
    jb.n = n;
    jb.k = (n + 31) & ~31;
    const int64_t mb = static_cast<int64_t>(kmax) * kmax * 8;
    for (int i = 0; i < kFp64Mats; ++i) jb.M[i] = reinterpret_cast<int64_t*>(slot + i * mb);
    for (int i = 0; i < kFp64Planes; ++i) jb.P[i] = slot + mats * mb + i * slice_bytes(kmax);
}
// The first bytes of a slot serve the cluster (kSlotHead); slice_job gets what follows.  The last hold the rows'
// squared lengths.
constexpr int64_t sums_bytes(int64_t k) { return 3 * 8 * k; }

// Adds the squared length of sixteen neighbouring entries of row r, half each of a lane pair (s: this lane's in units
// of 2^-24, the squares of at most eight entries of magnitude 2), to the row's sum: in integers, so that
// the sum is the same in every order.
__device__ __forceinline__ void add_length(unsigned long long* sums, int r, float s) {
    const unsigned int u = __float2uint_rn(s);
    const unsigned int both = u + __shfl_xor_sync(0xffffffffu, u, 1);
    if ((threadIdx.x & 1) == 0) atomicAdd(sums + r, static_cast<unsigned long long>(both));
}
// The squared length of eight fixed-point values in units of 2^-24 (their upper halves: units of 2^-30).
__device__ __forceinline__ float length8(const int64_t (&q)[8]) {
    float s = 0.0f;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const float x = static_cast<float>(static_cast<int>(q[i] >> 32));
        s = fmaf(x, x, s);
    }
    return s * 0x1p-36f;
}

__device__ __forceinline__ int64_t ld1(const int64_t* p) { return __ldcg(reinterpret_cast<const long long*>(p)); }

__device__ __forceinline__ unsigned long long cta_max_u64(unsigned long long v, SliceScalars* ss) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long w = __shfl_xor_sync(0xffffffffu, v, o);
        v = w > v ? w : v;
    }
    __syncthreads();
    if ((threadIdx.x & 31) == 0) ss->u[threadIdx.x >> 5] = v;
    __syncthreads();
    v = 0;
    for (int w = 0; w < kSliceWarps; ++w) v = ss->u[w] > v ? ss->u[w] : v;
    return v;
}

__device__ __forceinline__ unsigned long long warp_sum_u64(unsigned long long v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

__device__ __forceinline__ uint64_t abs_fixed(int64_t x) { return static_cast<uint64_t>(x < 0 ? -x : x); }

// What the following products keep: the weights up to 8 or 9, and the chunks of one accumulation.
__device__ __forceinline__ void set_accumulation(SliceShared* sh, int weights, int kpart) {
    __syncthreads();
    if (threadIdx.x == 0) {
        sh->weights = weights;
        sh->kpart = kpart;
    }
    __syncthreads();
}

// Submatrices whose shortest row (2-norm) is below kGraded times the longest go to the FP64 kernels (k_ns_graded.cu).
// The fixed point here holds an entry to 2^-57 of the longest row, floating point to 2^-53 of itself: for A = D S0 D, S0
// well conditioned, the relative error of the roots and of the sign grows as 1 / d^2 in the one (d the smallest entry
// of D) and not at all in the other.  An emulation of both (n = 16): at a ratio of the rows of 1, 1/5, 1/10, 1/20 and
// 1/100 the roots' error is 5e-17, 1e-16, 2e-16, 3e-16 and 2e-15 in fixed point, 2e-16 .. 6e-16 in FP64; the sign's
// 6e-17, 1e-16, 3e-16, 1e-15 and 2e-14, 3e-16 .. 1e-15 in FP64.  They cross between 1/10 and 1/20, so
// from 1/8 on none is further off than in FP64.  (The water-like systems' rows: 0.6 and more.)
constexpr float kGraded = 1.0f / 8.0f;

// Puts block column j on the list; one thread of a cluster calls it.
__device__ __forceinline__ void list_graded(GradedList* list, int j) { list->column[atomicAdd(&list->count, 1)] = j; }

// The cluster's sums of squared lengths (SliceJob::sums): cleared a phase before they are added to and a phase after
// every CTA has read them; the largest and the smallest of n of them.
__device__ __forceinline__ void clear_sums(unsigned long long* sums, int count) {
    for (int r = cluster_rank() * kSliceThreads + threadIdx.x; r < count; r += cluster_size() * kSliceThreads) __stcg(sums + r, 0ull);
}
__device__ __forceinline__ unsigned long long largest_sum(const unsigned long long* sums, int n, SliceScalars* ss) {
    unsigned long long m = 0;
    for (int r = threadIdx.x; r < n; r += kSliceThreads) m = max(m, __ldcg(sums + r));
    return cta_max_u64(m, ss);
}
__device__ __noinline__ bool sums_graded(const unsigned long long* sums, int n, SliceScalars* ss) {
    const unsigned long long most = largest_sum(sums, n, ss);
    unsigned long long m = 0;
    for (int r = threadIdx.x; r < n; r += kSliceThreads) m = max(m, ~__ldcg(sums + r));
    return static_cast<float>(~cta_max_u64(m, ss)) < kGraded * kGraded * static_cast<float>(most);
}

// The bits of entries (r, c .. c + 7) of a symmetric matrix of doubles (read along its rows), zero past n.
__device__ __forceinline__ void load_bits(const double* __restrict__ src, int ld, int n, int r, int c, int64_t (&v)[8]) {
#pragma unroll
    for (int i = 0; i < 8; ++i) v[i] = r < n && c + i < n ? __double_as_longlong(src[static_cast<int64_t>(c + i) * ld + r]) : 0;
}

// The elementwise passes between products (each a function of its own, so that its registers are
// its own: what the callers keep across it lies on the stack, not what its loop works on).

// The symmetric n x n matrix src - mu I, times f 2^-e, into M and the planes (see to_fixed).  The rows' squared
// lengths are added to sums, in units of 2^-48 (they may all be short: f 2^-e brings a bound of the eigenvalues to 1).
__device__ __noinline__ bool pass_source(const double* __restrict__ src, int ld, double mu, int e, uint64_t f, int64_t* M, uint8_t* planes, int n,
                                         int k, unsigned long long* sums = nullptr) {
    bool bad = false;
    slice_pass<1>(k, k, planes, [&](int r, int c, int64_t (&v)[1][8]) { load_bits(src, ld, n, r, c, v[0]); },
                  [&](int r, int c, const int64_t (&v)[1][8], int64_t (&q)[8]) {
#pragma unroll
                      for (int i = 0; i < 8; ++i) {
                          double x = __longlong_as_double(v[0][i]);
                          if (mu != 0.0 && r == c + i && r < n) x -= mu;
                          q[i] = to_fixed(x, e, f, bad);
                      }
                      st8(M, k, r, c, q);
                      if (sums) {
                          float s = length8(q);
                          s += __shfl_xor_sync(0xffffffffu, s, 1);
                          if ((threadIdx.x & 1) == 0) atomicAdd(sums + r, static_cast<unsigned long long>(s * 0x1p24f));
                      }
                  });
    return bad;
}

// The mean of an n x n matrix X and its transpose into M and the planes: a bulk phase's last iterate, which is
// symmetric up to that phase's rounding only (about 1e-7), while the products here take their factors
// for symmetric.
__device__ __noinline__ bool pass_iterate(const double* __restrict__ src, int ld, int64_t* M, uint8_t* planes, int n, int k) {
    bool bad = false;
    slice_pass<2>(k, k, planes,
                  [&](int r, int c, int64_t (&v)[2][8]) {
                      load_bits(src, ld, n, r, c, v[0]);
#pragma unroll
                      for (int i = 0; i < 8; ++i)
                          v[1][i] = r < n && c + i < n ? __double_as_longlong(src[static_cast<int64_t>(r) * ld + c + i]) : 0;
                  },
                  [&](int r, int c, const int64_t (&v)[2][8], int64_t (&q)[8]) {
#pragma unroll
                      for (int i = 0; i < 8; ++i) {
                          const int64_t x = to_fixed(__longlong_as_double(v[0][i]), 0, 0, bad);
                          const int64_t y = to_fixed(__longlong_as_double(v[1][i]), 0, 0, bad);
                          q[i] = (x >> 1) + (y >> 1);
                      }
                      st8(M, k, r, c, q);
                  });
    return bad;
}

// W = I - f S 2^up (f = 0: 1) to its digits; returns this thread's share of ||I - S 2^up||_F^2 in units of 2^-76.
// sums (with f = 0): the rows' squared lengths are added to it, far too long where an entry of S 2^up is above 1 (by
// more than rounding), of which the difference may not fit.
__device__ __noinline__ float pass_residual(const int64_t* S, uint8_t* planes, int n, int k, int up, uint64_t f,
                                            unsigned long long* sums = nullptr) {
    float r2 = 0.0f;
    const uint64_t most = static_cast<uint64_t>(kFixedOne + (kFixedOne >> 8)) >> up;
    slice_pass<1>(k, k, planes, [&](int r, int c, int64_t (&v)[1][8]) { ld8(S, k, r, c, v[0]); },
                  [&](int r, int c, const int64_t (&v)[1][8], int64_t (&q)[8]) {
                      float row = 0.0f;
                      uint64_t top = 0;
#pragma unroll
                      for (int i = 0; i < 8; ++i) {
                          const int64_t one = r == c + i && r < n ? kFixedOne : 0, s = v[0][i] << up;
                          const float d = fixed_float(one - s);
                          r2 = fmaf(d, d, r2);
                          row = fmaf(d, d, row);
                          top = max(top, abs_fixed(v[0][i]));
                          q[i] = one - (f ? fixed_mul(s, f) : s);
                      }
                      if (sums) add_length(sums, r, top > most ? 0x1p28f : fminf(row * 0x1p-52f, 0x1p28f));
                  });
    return r2;
}

// X <- f (X + 1/2 S) (f = 0: 1), and its digits; the rows' squared lengths are added to sums.
__device__ __noinline__ void pass_update(int64_t* X, const int64_t* S, uint8_t* planes, int k, uint64_t f, unsigned long long* sums = nullptr) {
    slice_pass<2>(k, k, planes,
                  [&](int r, int c, int64_t (&v)[2][8]) {
                      ld8(X, k, r, c, v[0]);
                      ld8(S, k, r, c, v[1]);
                  },
                  [&](int r, int c, const int64_t (&v)[2][8], int64_t (&q)[8]) {
#pragma unroll
                      for (int i = 0; i < 8; ++i) {
                          q[i] = v[0][i] + (v[1][i] >> 1);
                          if (f) q[i] = fixed_mul(q[i], f);
                      }
                      st8(X, k, r, c, q);
                      if (sums) add_length(sums, r, length8(q));
                  });
}

// Z <- 3/2 I - 1/2 (Y - 1/2 S); the rows' squared lengths are added to sums.
__device__ __noinline__ void pass_first_root(const int64_t* Y, const int64_t* S, int64_t* Z, int n, int k, unsigned long long* sums) {
    slice_pass<2>(k, k, nullptr,
                  [&](int r, int c, int64_t (&v)[2][8]) {
                      ld8(Y, k, r, c, v[0]);
                      ld8(S, k, r, c, v[1]);
                  },
                  [&](int r, int c, const int64_t (&v)[2][8], int64_t (&q)[8]) {
#pragma unroll
                      for (int i = 0; i < 8; ++i)
                          q[i] = (r == c + i && r < n ? kFixedOne + (kFixedOne >> 1) : 0) - ((v[0][i] - (v[1][i] >> 1)) >> 1);
                      st8(Z, k, r, c, q);
                      add_length(sums, r, length8(q));
                  });
}

// diag I +- f S 2^shift (f = 0: 1) to its digits, and to out when given.
__device__ __noinline__ void pass_affine(const int64_t* S, int64_t* out, uint8_t* planes, int n, int k, int64_t diag, bool minus, int shift,
                                         uint64_t f) {
    slice_pass<1>(k, k, planes, [&](int r, int c, int64_t (&v)[1][8]) { ld8(S, k, r, c, v[0]); },
                  [&](int r, int c, const int64_t (&v)[1][8], int64_t (&q)[8]) {
#pragma unroll
                      for (int i = 0; i < 8; ++i) {
                          // (modulo 2^64: 2 E of the Fermi form may be 2, one unit past the range, before I - 2 E)
                          int64_t x = shift >= 0 ? static_cast<int64_t>(static_cast<uint64_t>(v[0][i]) << shift) : v[0][i] >> min(-shift, 63);
                          if (f) x = fixed_mul(x, f);
                          const uint64_t d = r == c + i && r < n ? static_cast<uint64_t>(diag) : 0u;
                          q[i] = static_cast<int64_t>(minus ? d - static_cast<uint64_t>(x) : d + static_cast<uint64_t>(x));
                      }
                      if (out) st8(out, k, r, c, q);
                  });
}

// M <- 0.
__device__ __noinline__ void pass_zero(int64_t* M, int k) {
    slice_pass<1>(k, k, nullptr, [](int, int, int64_t (&)[1][8]) {},
                  [&](int r, int c, const int64_t (&)[1][8], int64_t (&q)[8]) {
#pragma unroll
                      for (int i = 0; i < 8; ++i) q[i] = 0;
                      st8(M, k, r, c, q);
                  });
}

// T <- (a T + b S) 2^up (a = 0: 1), and its digits.
__device__ __noinline__ void pass_mix(int64_t* T, const int64_t* S, uint8_t* planes, int k, uint64_t a, uint64_t b, int up) {
    slice_pass<2>(k, k, planes,
                  [&](int r, int c, int64_t (&v)[2][8]) {
                      ld8(T, k, r, c, v[0]);
                      ld8(S, k, r, c, v[1]);
                  },
                  [&](int r, int c, const int64_t (&v)[2][8], int64_t (&q)[8]) {
#pragma unroll
                      for (int i = 0; i < 8; ++i) q[i] = ((a ? fixed_mul(v[0][i], a) : v[0][i]) + fixed_mul(v[1][i], b)) << up;
                      st8(T, k, r, c, q);
                  });
}

// Digits of the transpose of columns c0 .. c0 + m - 1 of the k-row matrix A - B (B null: A; B's columns from
// 0), halved or shifted right: rows of an operand of `rows` x k.
__device__ __noinline__ void pass_transposed(const int64_t* A, const int64_t* B, int c0, int m, uint8_t* planes, int rows, int k, int shift) {
    slice_pass<1>(rows, k, planes, [&](int r, int c, int64_t (&v)[1][8]) {
#pragma unroll
        for (int i = 0; i < 8; ++i)
            v[0][i] = r < m ? (ld1(A + mat_at(k, c + i, c0 + r)) - (B ? ld1(B + mat_at(k, c + i, r)) : 0)) >> shift : 0;
    }, [](int, int, const int64_t (&v)[1][8], int64_t (&q)[8]) {
#pragma unroll
        for (int i = 0; i < 8; ++i) q[i] = v[0][i];
    });
}

// The symmetric source matrix A = src - mu I (n x n, leading dimension ld) in fixed point, A 2^-e, into M and
// the planes P.  The power of two brings the largest 2-norm of a row into (1/2, 1] (so that the
// products are exact and use all digits); kIterate: src is a bulk phase's iterate, made symmetric, e = 0.  bound: no entry is larger (0:
// not known).  Returns e; a value that is not finite sets ss->bad, and rows of very different size set ss->graded (but
// for kFactor, whose rows have been looked at): nothing is loaded then.
enum { kSource, kIterate, kFactor };
__device__ __noinline__ int load_fixed(const double* __restrict__ src, int ld, double mu, double bound, const SliceJob& jb, int64_t* M, uint8_t* P,
                          int kind, SliceShared* sh, SliceScalars* ss) {
    const bool iterate = kind == kIterate;
    const int n = jb.n, k = jb.k, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    auto entry = [&](int r, int c) -> double {
        const double v = src[static_cast<int64_t>(r) * ld + c];
        return r == c && mu != 0.0 ? v - mu : v;
    };
    const int ranks = cluster_size(), rank = cluster_rank();
    int e = 0;
    bool graded = false;
    if (threadIdx.x == 0) ss->bad = ss->graded = 0;
    if (!iterate) {
        uint32_t top = static_cast<uint32_t>(__double2hiint(bound)) & 0x7fffffffu;
        if (top == 0) {  // high words order like the magnitudes
            for (int r = warp + rank * kSliceWarps; r < n; r += ranks * kSliceWarps)
#pragma unroll 4
                for (int c = lane; c < n; c += 32) top = max(top, static_cast<uint32_t>(__double2hiint(entry(r, c))) & 0x7fffffffu);
            top = cluster_max(static_cast<uint32_t>(cta_max_u64(top, ss)), reinterpret_cast<uint32_t*>(jb.scratch) + 24);
        }
        const int ex = static_cast<int>(top >> 20);
        if (ex == 0x7ff) {
            __syncthreads();
            if (threadIdx.x == 0) ss->bad = 1;
            __syncthreads();
            return 0;
        }
        const int e0 = ex - 1022;  // |A| < 2^e0
        auto scaled = [&](double v) -> float {  // v 2^-e0, 0 below 2^-122
            const int hi = __double2hiint(v), ev = (hi >> 20) & 0x7ff, ef = ev - e0;
            return ev > 0 && ef > 900 ? d2f_rn(__hiloint2double((hi & 0x800fffff) | (ef << 20), __double2loint(v))) : 0.0f;
        };
        float worst = 0.0f, least = INFINITY;
        for (int r = 2 * (warp + rank * kSliceWarps); r < n; r += 2 * ranks * kSliceWarps) {
            const int r1 = min(r + 1, n - 1);
            float a0 = 0.0f, a1 = 0.0f;
#pragma unroll 4
            for (int c = lane; c < n; c += 32) {
                const float x = scaled(entry(r, c)), y = scaled(entry(r1, c));
                a0 = fmaf(x, x, a0);
                a1 = fmaf(y, y, a1);
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                a0 += __shfl_xor_sync(0xffffffffu, a0, o);
                a1 += __shfl_xor_sync(0xffffffffu, a1, o);
            }
            worst = fmaxf(worst, fmaxf(a0, a1));
            least = fminf(least, fminf(a0, a1));
        }
        // the largest, and the smallest by the largest complement (non-negative floats order like their bits)
        worst = cta_max(worst, sh);
        uint32_t rest = static_cast<uint32_t>(cta_max_u64(~__float_as_uint(least), ss));
        if (ranks > 1) {
            uint32_t* const ex = reinterpret_cast<uint32_t*>(jb.scratch);
            if (threadIdx.x == 0) {
                __stcg(ex + 8 + rank, __float_as_uint(worst));
                __stcg(ex + 56 + rank, rest);
            }
            phase_sync();
            for (int r = 0; r < ranks; ++r) {
                worst = fmaxf(worst, __uint_as_float(__ldcg(ex + 8 + r)));
                rest = max(rest, __ldcg(ex + 56 + r));
            }
        }
        graded = kind == kSource && __uint_as_float(~rest) < kGraded * kGraded * worst;
        e = e0 + (worst > 0.0f ? static_cast<int>(ceilf(0.5f * log2f(worst * 1.001f))) : 0);
    }
    __syncthreads();
    if (graded) {
        if (threadIdx.x == 0) ss->graded = 1;
        __syncthreads();
        return e;
    }
    const bool own_bad = iterate ? pass_iterate(src, ld, M, P, n, k) : pass_source(src, ld, mu, e, 0, M, P, n, k);
    const bool bad = cluster_sum(own_bad ? 1.0f : 0.0f, sh, jb.scratch) > 0.0f;
    if (bad) ss->bad = 1;
    __syncthreads();
    return e;
}

// The learned bound of a submatrix for sign_steps: the initial scaling b_j of X0 = A / b_j, the
// predicted smallest |eigenvalue| of A / b_j (negative: none) and the fallback counter.
struct SignModel {
    double b, dhat;
    int* fallbacks;
};
// What the first product gives: the largest row sum of |X0^2| and the factor c of the first step.
struct SignBound {
    double rmax, c;
};

// For the symmetric non-negative-bounded Y = S: the largest row sum of |Y| (every thread), and the smaller
// max_r (|Y| w)_r / w_r of two power steps from the row sums (thread 0; 0 without any).  The CTAs of a
// cluster take 32 rows each in turn and exchange the sums at `exchange`.  Memory there: 3 k values for that, and past
// kBoundSharedRows rows two vectors of k values for each CTA, which lie in the stage area below.
// (Held there for any k, they ran past its end from k = 13,472 on.)
constexpr int kBoundSharedRows = 2048;
static_assert(2 * 8 * kBoundSharedRows <= kSliceStages * kSliceStageBytes, "the two vectors fit the stage area");
static_assert((3 + 2 * 8) * 8 * kBoundSharedRows <= slice_bytes(kBoundSharedRows), "a matrix's planes hold the vectors of eight CTAs");
__device__ __noinline__ void first_bound(const int64_t* S, int n, int k, SliceShared* sh, SliceScalars* ss, unsigned long long* exchange,
                                         double& row_max, double& best) {
    const int ranks = cluster_size(), rank = cluster_rank();
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    unsigned long long* wv = k <= kBoundSharedRows ? reinterpret_cast<unsigned long long*>(sh->smem)
                                                   : exchange + static_cast<int64_t>(3 + 2 * rank) * k;  // row sums, then weights
    unsigned long long* av = wv + k;
    // entries are at most 1 (2^62): the sums of k of them, below in units of up to 2^-51, stay below 2^64
    const int cut = k <= 4096 ? 12 : 16;
    // v complete in every CTA of the cluster; the maximum (m: of the CTA's own rows)
    auto share = [&](unsigned long long* v, unsigned long long m) {
        if (ranks > 1) {
            __syncthreads();
            for (int r = tid; r < n; r += kSliceThreads)
                if ((r >> 5) % ranks == rank) __stcg(exchange + r, v[r]);
            phase_sync();
            for (int r = tid; r < n; r += kSliceThreads)
                if ((r >> 5) % ranks != rank) {
                    v[r] = __ldcg(exchange + r);
                    m = max(m, v[r]);
                }
            exchange += k;
        }
        return cta_max_u64(m, ss);
    };
    // row sums of |Y| in units of 2^(cut - 62)
    unsigned long long m = 0;
    for (int r = 2 * (warp + rank * kSliceWarps); r < n; r += 2 * ranks * kSliceWarps) {  // Y is symmetric: two columns at a time
        const longlong2* y = reinterpret_cast<const longlong2*>(S) + static_cast<int64_t>(r >> 1) * k;
        unsigned long long a0 = 0, a1 = 0;
#pragma unroll 4
        for (int c = lane; c < k; c += 32) {
            const longlong2 v = __ldcg(y + c);
            a0 += abs_fixed(v.x) >> cut;
            a1 += abs_fixed(v.y) >> cut;
        }
        a0 = warp_sum_u64(a0);
        a1 = warp_sum_u64(a1);
        if (lane == 0) {
            wv[r] = a0;
            wv[r + 1] = a1;
        }
        m = max(m, max(a0, a1));
    }
    m = share(wv, m);
    row_max = ldexp(static_cast<double>(m), cut - 62);
    best = 0.0;  // of the power steps (every row's quotient; 0: none)
    for (int pass = 0; pass < 2 && m > 0; ++pass) {
        // weights: any multiple of w serves; the largest into [2^62, 2^63), at least one unit
        const int up = __clzll(static_cast<long long>(m)) - 1;
        for (int r = tid; r < k; r += kSliceThreads) {
            const unsigned long long w = r < n ? wv[r] : 0ull;
            wv[r] = max(up >= 0 ? w << up : w >> -up, 1ull);
        }
        __syncthreads();
        m = 0;
        for (int r = 2 * (warp + rank * kSliceWarps); r < n; r += 2 * ranks * kSliceWarps) {
            const longlong2* y = reinterpret_cast<const longlong2*>(S) + static_cast<int64_t>(r >> 1) * k;
            unsigned long long a0 = 0, a1 = 0;  // (|Y| w)_r, w in units of 2^-63, in units of 2^(cut - 63)
#pragma unroll 4
            for (int c = lane; c < k; c += 32) {  // (zero past n)
                const longlong2 v = __ldcg(y + c);
                const unsigned long long w = wv[c] << 1;
                a0 += __umul64hi(abs_fixed(v.x) << 1, w) >> cut;
                a1 += __umul64hi(abs_fixed(v.y) << 1, w) >> cut;
            }
            a0 = warp_sum_u64(a0);
            a1 = warp_sum_u64(a1);
            if (lane == 0) {
                av[r] = a0;
                av[r + 1] = a1;
            }
            m = max(m, max(a0, a1));
        }
        m = share(av, m);
        double q = 0.0;
        if (32 * warp < n) {  // FP64 divisions only on the warps that hold rows
            for (int r = tid; r < n; r += kSliceThreads) q = fmax(q, static_cast<double>(av[r]) / static_cast<double>(wv[r]));
            q = warp_max(q);
        }
        __syncthreads();
        if (lane == 0) ss->d[warp] = q;
        for (int r = tid; r < n; r += kSliceThreads) wv[r] = av[r];
        __syncthreads();
        if (tid == 0) {
            for (int w = 1; w < kSliceWarps; ++w)
                if (ss->d[w] > q) q = ss->d[w];
            q = ldexp(q, cut);
            best = pass == 0 ? q : fmin(best, q);
        }
    }
    phase_sync();              // `exchange` is the caller's again: no CTA of the cluster still reads it
    fence_proxy_async_smem();  // the stages are the copies' again
}

// Newton-Schulz steps on X = M[0] (digits in P[0]; A = X 2^e) until the residual is <= tau (returns
// the number of steps; conv, bad).  plain_steps > 0: exactly that many plain steps.  M[1] takes the
// products, P[1] the digits of W.
//
// The first product bounds the spectrum (as in the tensor-core kernel): with Y = X0^2, rho(X0)^2 =
// rho(Y) <= rho(|Y|) <= max_r (|Y| w)_r / w_r for any positive w (Collatz-Wielandt): w = 1 (the
// largest row sum) and two power steps of |Y| from it, in integers; the iteration continues from
// c X0, c = 1.2 / s.  A scaled step X' = p(a X), p(x) = x (3 - x^2) / 2, is a (X + 1/2 X W), W =
// I - a^2 X^2.
__device__ int sign_steps(SliceShared* sh, const SliceJob& jb, int e, int max_iter, float tau, int plain_steps, const SignModel* model,
                          SignBound* bound_out, SliceScalars* ss, bool& conv, bool& bad) {
    const int n = jb.n, k = jb.k, tid = threadIdx.x;
    int64_t *X = jb.M[0], *S = jb.M[1];
    conv = bad = false;
    int done = 0;
    if (tid == 0) ss->lsch = 1.0;
    const int limit = plain_steps > 0 ? plain_steps : max_iter;
    for (int it = 0; it < limit; ++it) {
        slice_product(sh, jb.P[0], jb.P[0], k, k, S, true);
        if (*static_cast<volatile int*>(&sh->abort)) break;
        if (it == 0 && plain_steps == 0) {
            double row_max, best;
            first_bound(S, n, k, sh, ss, reinterpret_cast<unsigned long long*>(jb.P[1]), row_max, best);
            if (tid == 0) {
                // s >= rho(X0); the model's rules are stated for A / b_j = X0 / phi
                const double rmax = row_max;
                const double smax = sqrt(fmin(best, rmax) * (1.0 + 1e-12));
                double c = smax > 0.0 ? 1.2 / smax : 1.0, lsch = 1.0;
                if (model && smax > 0.0) {  // same rule as the tensor-core kernel
                    const double phi = ldexp(model->b, -e), s1 = smax / phi;
                    double scale = 1.2 / s1;
                    const bool gap = model->dhat > 0.0;
                    if (gap ? model->dhat <= s1 : s1 <= 1.7) {
                        if (gap) {  // the scaled schedule from l0 = dhat / s
                            const double l0 = model->dhat / s1, a0 = ns_scale(l0);
                            scale = a0 / s1;
                            lsch = ns_next_lower(a0, l0);
                        } else {
                            scale = fmax(1.0, scale);
                        }
                    } else {
                        if (cluster_rank() == 0) atomicAdd(model->fallbacks, 1);
                    }
                    c = scale / phi;
                }
                bound_out->rmax = rmax;
                bound_out->c = c;
                ss->lsch = lsch;
                ss->f1 = fixed_factor(c);
                ss->f2 = fixed_factor(c * c);
                ss->stop = 0;
            }
        } else if (tid == 0) {
            const double l = ss->lsch;
            ss->f1 = ss->f2 = 0;
            ss->stop = 1;
            if (l < 1.0) {  // the scaled schedule
                const double f = ns_scale(l);
                ss->lsch = ns_next_lower(f, l);
                ss->f1 = fixed_factor(f);
                ss->f2 = fixed_factor(f * f);
                ss->stop = f - 1.0 <= 2e-6;
            }
        }
        __syncthreads();
        const uint64_t f1 = ss->f1, f2 = ss->f2;
        // W = I - a^2 X^2 to its digits; the residual ||I - X^2||_F
        float r2 = pass_residual(S, jb.P[1], n, k, 0, f2);
        r2 = cluster_sum(r2 * 0x1p-76f, sh, jb.scratch);
        slice_product(sh, jb.P[0], jb.P[1], k, k, S, true);
        if (*static_cast<volatile int*>(&sh->abort)) break;
        done = it + 1;
        bad = !isfinite(r2);
        bool last = bad || done == limit;
        if (plain_steps == 0 && it > 0 && sqrtf(r2) <= tau) {
            // stop after this step unless it was a scaled step whose factor moves converged
            // eigenvalues off 1 (p(a) ~ 1 - 1.5 (a - 1)^2): then plain steps from here
            if (ss->stop) {
                conv = last = true;
            } else {
                __syncthreads();
                if (tid == 0) ss->lsch = 1.0;
            }
        }
        pass_update(X, S, last ? nullptr : jb.P[0], k, f1);
        if (last) break;
    }
    return done;
}

// Largest 2-norm of a column of M, squared.  The CTAs of a cluster take the columns in turn; the barrier of
// their maximum also orders every read of M before what follows (the callers change M in place).
__device__ __noinline__ float column_norm2(const SliceJob& jb, const int64_t* M, SliceShared* sh) {
    const int n = jb.n, k = jb.k, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int ranks = cluster_size(), rank = cluster_rank();
    float worst = 0.0f;
    for (int c = 2 * (warp + rank * kSliceWarps); c < n; c += 2 * ranks * kSliceWarps) {
        const longlong2* m = reinterpret_cast<const longlong2*>(M) + static_cast<int64_t>(c >> 1) * k;
        float a0 = 0.0f, a1 = 0.0f;
#pragma unroll 4
        for (int r = lane; r < k; r += 32) {
            const longlong2 v = __ldcg(m + r);
            const float x = static_cast<float>(static_cast<int>(v.x >> 32)), y = static_cast<float>(static_cast<int>(v.y >> 32));
            a0 = fmaf(x, x, a0);
            a1 = fmaf(y, y, a1);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            a0 += __shfl_xor_sync(0xffffffffu, a0, o);
            a1 += __shfl_xor_sync(0xffffffffu, a1, o);
        }
        worst = fmaxf(worst, fmaxf(a0, a1));
    }
    worst = cta_max(worst, sh);
    return __uint_as_float(cluster_max(__float_as_uint(worst), reinterpret_cast<uint32_t*>(jb.scratch) + 32)) * 0x1p-60f;
}

// The sign iteration of the Eq. 12 block matrix [[0, A], [I, 0]] written per block (the coupled
// Newton-Schulz iteration): R = I - Z Y, Y <- Y + 1/2 Y R, Z <- Z + 1/2 R Z from Y = A / b (eigenvalues in
// (0, 1]) and Z = I; Y -> (A / b)^1/2, Z -> (A / b)^-1/2.  The residual ||Z Y - I||_F comes with the
// first product; the stopping rule is the sign iteration's.  src is A (leading dimension ld), b >= its
// largest eigenvalue.  Y ends in M[0] (digits P[0]), Z in M[1] (digits P[1]) in units of 2^(ez - 62); M[2]
// takes the products, P[2] the digits of R.  Every matrix is a polynomial of A, so the products are
// symmetric.  The first step needs one product (Z = I), the last only that of the wanted root.
//
// Positive definiteness.  For a positive definite A the eigenvalues of Y and R lie in [0, 1], so no row of them is
// longer than 1 and no entry of Z Y is larger, and a step lengthens no row of Z by more than 3/2 (Z's are kept
// below 1 by its exponent).  The integers would wrap where floating point overflows, and the iteration could then
// converge to a root of another matrix.  So the passes add up the rows' squared lengths, and a matrix whose
// rows are too long enters no product: with rows of at most 1 in both factors no entry of a product leaves
// the integers' range, nor does X + 1/2 X R, and nothing wraps before it is seen.  A negative eigenvalue -t of Z Y
// grows from step to step (t (3 + t)^2 / 4 > 2.25 t) until the rows of R, which hold its 1 + t, are too long.
//
// Returns the number of steps, -1 for rows of very different size (kGraded); with want_z ss->graded tells whether Z's are.
__device__ int coupled_steps(SliceShared* sh, const SliceJob& jb, const double* __restrict__ src, int ld, double b, int max_iter, float tau,
                             bool want_y, bool want_z, int& ez, SliceScalars* ss, bool& conv, bool& bad) {
    const int n = jb.n, k = jb.k;
    int64_t *Y = jb.M[0], *Z = jb.M[1], *S = jb.M[2];
    unsigned long long *row_r = jb.sums, *row_y = row_r + k, *row_z = row_y + k;  // squared lengths in units of 2^-24
    auto longest = [&](const unsigned long long* sums) { return static_cast<float>(largest_sum(sums, n, ss)) * 0x1p-24f; };
    constexpr float kLongest = 1.002f;  // of a length squared that is at most 1 (its squares are rounded)
    clear_sums(row_r, 3 * k);
    phase_sync();
    conv = bad = false;
    ez = 0;
    int done = 0;
    // 1 / b as a 64-bit fraction in [1/2, 1) times a power of two
    const double inv = 1.0 / b;
    const uint64_t ib = static_cast<uint64_t>(__double_as_longlong(inv));
    const uint64_t f = ((ib & 0xfffffffffffffull) | 0x10000000000000ull) << 11;
    const int e = 1022 - static_cast<int>((ib >> 52) & 0x7ff);
    bool off = !(b > 0.0) || !isfinite(inv) || inv == 0.0;
    off |= pass_source(src, ld, 0.0, e, f, Y, jb.P[0], n, k, row_z);
    const bool graded = sums_graded(row_z, n, ss);
    if (cluster_sum(off ? 1.0f : 0.0f, sh, jb.scratch) > 0.0f) {
        bad = true;
        return 0;
    }
    if (graded) return -1;
    for (int it = 0; it < max_iter; ++it) {
        if (it > 0) {
            slice_product(sh, jb.P[1], jb.P[0], k, k, S, true);  // Z Y
            if (*static_cast<volatile int*>(&sh->abort)) break;
        }
        clear_sums(row_y, 2 * k);
        float r2 = pass_residual(it > 0 ? S : Y, jb.P[2], n, k, ez, 0, row_r);
        r2 = cluster_sum(r2 * 0x1p-76f, sh, jb.scratch);
        done = it + 1;
        if (longest(row_r) > kLongest) {
            bad = true;
            break;
        }
        conv = it > 0 && sqrtf(r2) <= tau;
        if (!conv || want_y) {
            slice_product(sh, jb.P[0], jb.P[2], k, k, S, true);  // Y R
            if (*static_cast<volatile int*>(&sh->abort)) break;
            clear_sums(row_r, k);
            pass_update(Y, S, jb.P[0], k, 0, row_y);
        }
        if (!conv || want_z) {
            if (it > 0) {
                slice_product(sh, jb.P[2], jb.P[1], k, k, S, true);  // R Z
                if (*static_cast<volatile int*>(&sh->abort)) break;
            }
            // Z' = Z + 1/2 R Z; from Z = I: I + 1/2 R = 3/2 I - 1/2 Y0, where Y now holds Y0 + 1/2 Y0 R and S = Y0 R
            if (it > 0) pass_update(Z, S, nullptr, k, 0, row_z);
            else pass_first_root(Y, S, Z, n, k, row_z);
            const float z = longest(row_z);
            const int shift = z > 1.0f ? 1 : 0;
            ez += shift;
            if (z > 2.25f * kLongest || longest(row_y) > kLongest || ez > 40) {
                bad = true;
                conv = false;
                break;
            }
            pass_affine(Z, shift ? Z : nullptr, jb.P[1], n, k, 0, false, -shift, 0);
        }
        if (conv) break;
    }
    if (conv && want_z) {
        const bool z_graded = sums_graded(row_z, n, ss);
        if (threadIdx.x == 0) ss->graded = z_graded;
        __syncthreads();
    }
    return done;
}

// The finite-temperature Fermi function F = (I + exp(beta A))^-1 = 1/2 (I - tanh(beta A / 2)) of a
// symmetric A (src, leading dimension ld; g >= its spectral radius), in products only:
//   B = beta A / 2^(m + 1) with m such that ||B|| <= 1/16;
//   T = tanh(B) by its odd Taylor series to degree 11 (the next term is below 1e-18 there);
//   m doublings tanh(2x) = 2 tanh(x) / (1 + tanh(x)^2): with E = T^2 (eigenvalues in [0, 1]) and
//   Q = I - 2 E the linear approximation V0 = 2/3 I + 2/9 Q of (I + E)^-1 leaves the residual
//   I - (I + E) V0 = Q^2 / 9 = K, so T' = 2 T V0 (I + K) (I + K^2) (I + K^4) (I + K^8) (I + K^16)
//   to 1e-30: twelve products a doubling;
//   F = 1/2 (I - T).
// A doubling at most doubles an error in T (m = 11 at beta g = 150).  T is kept as T 2^t with the
// largest t for which its norm bound min(1, 2^doublings / 16) stays below 1.  The result's T 2^t is in
// M[0] (units of 2^-62), t in ss->e; M[1] takes the products.  Returns the number of products, -1 for rows
// of very different size (kGraded).
__device__ int fermi_tanh(SliceShared* sh, const SliceJob& jb, const double* __restrict__ src, int ld, double g, double beta, SliceScalars* ss,
                          bool& bad) {
    const int n = jb.n, k = jb.k;
    int64_t *T = jb.M[0], *S = jb.M[1];
    uint8_t *PT = jb.P[0], *PK = jb.P[1], *PP = jb.P[2];
    bad = false;
    if (threadIdx.x == 0) ss->e = 0;
    int m = 0;
    double sc = 0.5 * beta * g;
    while (sc > 1.0 / 16.0 && m < 60) {
        sc *= 0.5;
        ++m;
    }
    // B 2^s with ||B 2^s|| <= 1: s = the exponent room of sc
    int s2 = 0;
    if (sc > 0.0)
        while (sc < 0.5 && s2 < 60) {
            sc *= 2.0;
            ++s2;
        }
    // A (beta / 2^(m + 1)) 2^s2 = A sc / g
    const double fac = sc / g;
    const uint64_t ib = static_cast<uint64_t>(__double_as_longlong(fac));
    const uint64_t f = ((ib & 0xfffffffffffffull) | 0x10000000000000ull) << 11;
    const int e = 1022 - static_cast<int>((ib >> 52) & 0x7ff);
    const bool zero = !(fac > 0.0);
    bool off = !isfinite(fac);
    bool graded = false;
    if (!zero && !off) {
        clear_sums(jb.sums, k);
        phase_sync();
        off = pass_source(src, ld, 0.0, e, f, T, PT, n, k, jb.sums);
        graded = sums_graded(jb.sums, n, ss);
    }
    if (cluster_sum(off ? 1.0f : 0.0f, sh, jb.scratch) > 0.0f) {
        bad = true;
        return 0;
    }
    if (zero) {  // (the slot holds what the submatrix before left)
        pass_zero(T, k);
        return 0;
    }
    if (graded) return -1;
    int nprod = 0;
    // wide: with the digit pairs of weight 9 (an error in T may double at every doubling; the products of
    // K enter it with factors of 1/9 and less)
    auto prod = [&](const uint8_t* a, const uint8_t* b, bool wide) {
        set_accumulation(sh, wide ? 8 : 7, wide ? 160 / 16 : kSliceK / 16);
        slice_product(sh, a, b, k, k, S, true);
        ++nprod;
        return *static_cast<volatile int*>(&sh->abort) == 0;
    };
    const double cs[6] = {1.0, -1.0 / 3.0, 2.0 / 15.0, -17.0 / 315.0, 62.0 / 2835.0, -1382.0 / 155925.0};
    auto fixed = [](double v) { return static_cast<int64_t>(v * 0x1p62); };
    // Y = B^2 (digits of Y 2^(2 s2)); P = c4 + c5 Y, then P <- c_i + P Y
    if (!prod(PT, PT, true)) return nprod;
    const int down = 2 * s2;
    const uint64_t c5 = fixed_factor(-cs[5]);
    const int64_t c4 = fixed(cs[4]);
    pass_affine(S, nullptr, PP, n, k, c4, true, -down, c5);
    pass_affine(S, nullptr, PK, n, k, 0, false, 0, 0);
    for (int i = 3; i >= 0; --i) {
        if (!prod(PP, PK, true)) return nprod;
        const int64_t ci = fixed(cs[i]);
        pass_affine(S, nullptr, PP, n, k, ci, false, -down, 0);
    }
    if (!prod(PT, PP, true)) return nprod;
    pass_affine(S, T, PT, n, k, 0, false, 0, 0);
    int t = s2;
    const uint64_t f23 = fixed_factor(2.0 / 3.0), f29 = fixed_factor(2.0 / 9.0);
    for (int d = 0; d < m; ++d) {
        // E = T^2 (S holds E 2^(2 t)), Q = I - 2 E
        if (!prod(PT, PT, true)) return nprod;
        const int dn = 2 * t;
        pass_affine(S, nullptr, PK, n, k, kFixedOne, true, 1 - dn, 0);
        // U = T V0 (times 2 when T 2^t has no exponent room left; else 2 T V0 has one less)
        if (!prod(PT, PK, true)) return nprod;
        const int up = t > 0 ? 0 : 1;
        t = t > 0 ? t - 1 : 0;
        pass_mix(T, S, PT, k, f23, f29, up);
        // K = Q^2 / 9 (digits of 9^j K^j: powers of Q^2), U <- U + U K^j for j = 1, 2, 4, 8, 16
        double w = 1.0 / 9.0;
        for (int j = 0; j < 5; ++j) {
            if (!prod(PK, PK, false)) return nprod;
            pass_affine(S, nullptr, PK, n, k, 0, false, 0, 0);
            if (!prod(PT, PK, false)) return nprod;
            pass_mix(T, S, PT, k, 0, fixed_factor(w), 0);
            w *= w;
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) ss->e = t;
    __syncthreads();
    return nprod;
}

// The symmetric matrix f M as doubles, row by row.
__device__ __noinline__ void store_scaled(const int64_t* M, int k, double f, double* __restrict__ out, int n, int ld) {
    for (int r = cluster_rank() * kSliceWarps + (threadIdx.x >> 5); r < n; r += cluster_size() * kSliceWarps)
        for (int c = threadIdx.x & 31; c < n; c += 32)  // row r is column r
            out[static_cast<int64_t>(r) * ld + c] = f * static_cast<double>(ld1(M + mat_at(k, c, r)));
}

// Gershgorin interval (lo, hi) of an n x n matrix held row by row.
__device__ double2 gershgorin_interval(const double* M, int n, int ld, double* scratch) {
    const int warp = threadIdx.x / 32, lane = threadIdx.x & 31;
    double lo = INFINITY, hi = -INFINITY;
    for (int r = warp; r < n; r += kSliceWarps) {
        double acc = 0.0;
        for (int c = lane; c < n; c += 32) acc += c == r ? 0.0 : fabs(M[static_cast<int64_t>(r) * ld + c]);
        acc = warp_sum(acc);
        const double d = M[static_cast<int64_t>(r) * ld + r];
        lo = fmin(lo, d - acc);
        hi = fmax(hi, d + acc);
    }
    if (lane == 0) {
        scratch[warp] = lo;
        scratch[32 + warp] = hi;
    }
    __syncthreads();
    double2 out = make_double2(INFINITY, -INFINITY);
    for (int w = 0; w < kSliceWarps; ++w) {
        out.x = fmin(out.x, scratch[w]);
        out.y = fmax(out.y, scratch[32 + w]);
    }
    __syncthreads();
    return out;
}

// The next submatrix of the CTA or cluster (largest first; every thread gets its place in the order): its
// own place first, then whichever is next when it is free.  (Claimed one ahead, 256 submatrices on 152
// SMs took 8 % longer: some SMs held two of the largest.)  Meanwhile the source of the submatrix that
// the launch is likely to reach next comes into L2.  shared_jobs: two words of the cluster, taken in turn: a
// submatrix may pass without a barrier of the cluster (one that is not finite), and then a CTA may still
// have to read its word when the first CTA writes the next one.
__device__ __forceinline__ int claim_job(int* counter, SliceScalars* ss, SubDesc* cur, int* shared_jobs, int round, int n_subs,
                                         const int32_t* order, const SubDesc* subs, const double* src) {
    __syncthreads();
    const int ranks = cluster_size(), clusters = gridDim.x / ranks;
    const bool leader = cluster_rank() == 0;
    int* const shared_job = shared_jobs + (round & 1);
    if (threadIdx.x == 0 && leader) {
        const int job = round == 0 ? blockIdx.x / ranks : clusters + atomicAdd(counter, 1);
        if (ranks > 1) __stcg(shared_job, job);
        ss->job = job;
        if (job + clusters < n_subs) {
            const SubDesc& s = subs[order[job + clusters]];
            const uint64_t bytes = static_cast<uint64_t>(s.n) * s.ld * sizeof(double);
            asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(src + s.t_off),
                         "r"(static_cast<uint32_t>(bytes < (8u << 20) ? bytes : (8u << 20)) & ~15u)
                         : "memory");
        }
    }
    if (ranks > 1) phase_sync();
    if (threadIdx.x == 0) {
        if (!leader) ss->job = __ldcg(shared_job);
        if (ss->job < n_subs) *cur = subs[order[ss->job]];
    }
    __syncthreads();
    return ss->job;
}

// The last cluster to run out of work resets the job counter for the next launch.
// A leader that gave up leaves its cluster no job to find.
__device__ __forceinline__ void release_jobs(int* counter, unsigned int* ticket, int* shared_jobs) {
    if (threadIdx.x == 0 && cluster_rank() == 0) {
        __stcg(shared_jobs, INT_MAX);
        __stcg(shared_jobs + 1, INT_MAX);
        __threadfence();
        if (atomicAdd(ticket, 1u) == gridDim.x / cluster_size() - 1) {
            *counter = 0;
            *ticket = 0u;
        }
    }
}

__device__ __forceinline__ uint8_t* slice_stages() {
    extern __shared__ uint8_t slice_smem_raw[];
    return reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(slice_smem_raw) + 1023) & ~uintptr_t(1023));
}

}  // namespace

// FORM: the sign iteration, the coupled iteration of the roots or the Fermi function (one kernel each:
// together their live values would not fit the registers).
enum { kFormSign, kFormRoots, kFormFermi };

template <int FORM>
__global__ void __launch_bounds__(kSliceThreads, 1) k_ns_fp64(const __grid_constant__ NsFp64Args a) {
    __shared__ SliceShared shared;
    __shared__ SliceScalars ss;
    __shared__ SignBound sb;
    __shared__ SubDesc s;
    __shared__ SliceJob jb;
    __shared__ double scratch[64];
    if (a.skip && *a.skip) return;
    SliceShared* const sh = &shared;
    int* ls_smem = reinterpret_cast<int*>(slice_stages());  // local block starts, between products only
    slices_begin(sh, slice_stages(), a.status);
    uint8_t* slot = a.ws + static_cast<int64_t>(blockIdx.x / cluster_size()) * a.slot_bytes;
    const bool lead = cluster_rank() == 0;  // writes the results
    for (int round = 0;; ++round) {
        const int job = claim_job(a.work_counter, &ss, &s, reinterpret_cast<int*>(slot + 64), round, a.n_subs, a.order, a.subs, a.Mc ? a.Mc : a.T);
        if (job >= a.n_subs || sh->abort) break;
        const int j = s.col;
        if (threadIdx.x == 0) {
            slice_job(jb, slot + kSlotHead, s.n, a.kmax, a.mats);
            jb.scratch = reinterpret_cast<float*>(slot);
            jb.sums = reinterpret_cast<unsigned long long*>(slot + a.slot_bytes - sums_bytes(a.kmax));
        }
        __syncthreads();
        const int n = s.n, k = jb.k;
        const double* T = a.T + s.t_off;
        bool conv = false, bad = false;
        int done = 0;
        if constexpr (FORM == kFormFermi) {
            done = fermi_tanh(sh, jb, T, s.ld, a.bound[j], a.beta, &ss, bad);
            if (sh->abort) break;
            if (done < 0) {
                if (threadIdx.x == 0 && lead) list_graded(a.graded, j);
                continue;
            }
            if (threadIdx.x == 0 && lead) {
                a.iters[j] = done;
                atomicAdd(a.work_n3, static_cast<unsigned long long>(n) * n * n * done);
                if (bad) atomicCAS(a.status, kOk, kErrNonfinite);
            }
            const int64_t* F = jb.M[0];
            const double fs = bad ? NAN : ldexp(1.0, -ss.e);
            auto frow = [&](int q, int i) -> double { return fs * from_fixed(ld1(F + mat_at(k, i, s.own + q))); };
            if (lead) finish_column(s, a.pv, a.H, a.D, a.partial, frow, ls_smem, scratch);  // 1/2 (I - T)
            fence_proxy_async_smem();
            continue;
        } else if constexpr (FORM == kFormRoots) {
            // f = A^-1/2, A^1/2 or A^-1 for a symmetric positive definite A = T_j - mu I
            int ez = 0;
            const double b = a.bound[j];
            done = coupled_steps(sh, jb, T, s.ld, b, a.max_iter, static_cast<float>(a.tau), a.function == kFnSqrt, a.function != kFnSqrt, ez,
                                 &ss, conv, bad);
            if (sh->abort) break;
            if (done < 0) {
                if (threadIdx.x == 0 && lead) list_graded(a.graded, j);
                continue;
            }
            if (threadIdx.x == 0 && lead) {
                a.iters[j] = done;
                atomicAdd(a.work_n3, static_cast<unsigned long long>(n) * n * n * done);
                if (bad) atomicCAS(a.status, kOk, kErrNonfinite);
                else if (!conv) atomicCAS(a.status, kOk, kErrNoconv);
            }
            // A^-1/2 = Z / sqrt(b), A^1/2 = sqrt(b) Y, A^-1 = Z Z / b (symmetric: row own + q is
            // column own + q)
            const int64_t* F = a.function == kFnSqrt ? jb.M[0] : jb.M[1];
            double fs = a.function == kFnSqrt ? sqrt(b) : ldexp(1.0 / sqrt(b), ez);
            if (a.function == kFnInv) {
                slice_product(sh, jb.P[1], jb.P[1], k, k, jb.M[2], true);
                if (sh->abort) break;
                F = jb.M[2];
                fs = ldexp(1.0 / b, 2 * ez);
            }
            if (bad) fs = NAN;
            auto frow = [&](int q, int i) -> double { return fs * from_fixed(ld1(F + mat_at(k, i, s.own + q))); };
            if (lead) finish_column(s, a.pv, a.H, a.D, a.partial, frow, ls_smem, scratch, false);
            fence_proxy_async_smem();
            continue;
        } else {
        // the sign iteration: on T_j - mu I, on M_j - mu I (non-orthogonal form: M_j = L_j A_H L_j from the
        // setup kernel), or FP64 finishing steps on a bulk phase's last iterate
        const double* src = a.Mc ? a.Mc + s.t_off : T;
        if (a.Mc) {  // its Gershgorin bound
            const int warp = threadIdx.x / 32, lane = threadIdx.x & 31;
            double rmax = 0.0;
            for (int r = warp; r < n; r += kSliceWarps) {
                double acc = 0.0;
                for (int c = lane; c < n; c += 32) acc += fabs(src[static_cast<int64_t>(r) * s.ld + c] - (r == c ? a.mu : 0.0));
                rmax = fmax(rmax, warp_sum(acc));
            }
            if (lane == 0) scratch[warp] = rmax;
            __syncthreads();
            if (threadIdx.x == 0) {
                double b = 0.0;
                for (int w = 0; w < kSliceWarps; ++w) b = fmax(b, scratch[w]);
                scratch[32] = b > 0.0 ? b : 1.0;
                if (lead) a.gersh[j] = scratch[32];
            }
            __syncthreads();
        }
        const bool finish = a.finish_iters > 0;
        const double gersh = a.Mc ? scratch[32] : a.gersh[j];
        SignModel model{a.bound[j], a.pred ? static_cast<double>(a.pred[2 * j + 1]) * gersh / a.bound[j] : -1.0, a.fallbacks};
        const int e = load_fixed(src, s.ld, a.Mc ? a.mu : 0.0, gersh, jb, jb.M[0], jb.P[0], finish ? kIterate : kSource, sh, &ss);
        bad = ss.bad != 0;
        if (!bad && (ss.graded || (a.Mc && a.root_graded[j]))) {  // (L is a factor of the result)
            if (threadIdx.x == 0 && lead) list_graded(a.graded, j);
            continue;
        }
        // with the learned bound W reaches a norm of 2, with a bulk phase's iterate X one of about 1.2
        set_accumulation(sh, 7, a.use_model || finish ? 160 / 16 : kSliceK / 16);
        if (!bad)
            done = sign_steps(sh, jb, e, a.max_iter, static_cast<float>(a.tau), a.finish_iters, a.use_model ? &model : nullptr, &sb, &ss, conv,
                              bad);
        if (sh->abort) break;
        if (threadIdx.x == 0 && lead) {
            if (finish) {
                a.iters[j] += done;
            } else {
                a.iters[j] = done;
                if (!bad || done > 0) {
                    // feature of the next snapshot: the Gershgorin bound of A^2, over G; and the
                    // effective bound of c X0
                    a.sq_ratio[j] = static_cast<float>(ldexp(sqrt(sb.rmax), e) / gersh);
                    a.bound[j] = ldexp(1.0 / sb.c, e);
                }
            }
            atomicAdd(a.work_n3, static_cast<unsigned long long>(n) * n * n * done);
            if (bad) atomicCAS(a.status, kOk, kErrNonfinite);
            else if (!conv && !finish) atomicCAS(a.status, kOk, kErrNoconv);
        }
        const int64_t* X = jb.M[0];
        if (a.Mc) {
            // P_j[:, own] = 1/2 L (I - X) L[:, own] = 1/2 L (W - X W), W = L[:, own] (rows own..
            // of the symmetric L): Eq. 14 with sign(A_S^-1 A_H - mu I) = L sign(M - mu I) L^-1
            // and A_S^-1 = L L.  Two products with the owner columns only: the digits of X in P[0], of L in
            // P[1], of W^T and then of 1/2 (W - X W)^T in P[2]; the products in M[1].
            set_accumulation(sh, 8, 160 / 16);
            pass_affine(X, nullptr, jb.P[0], n, k, 0, false, 0, 0);
            int64_t *L = jb.M[0], *U = jb.M[1];
            const int el = load_fixed(a.Lc + s.t_off, s.ld, 0.0, 0.0, jb, L, jb.P[1], kFactor, sh, &ss);
            const int w = s.bown <= 16 ? 16 : (s.bown + 31) & ~31;
            pass_transposed(L, nullptr, s.own, s.bown, jb.P[2], w, k, 0);
            slice_product(sh, jb.P[0], jb.P[2], k, w, U, false);
            if (sh->abort) break;
            pass_transposed(L, U, s.own, s.bown, jb.P[2], w, k, 1);
            slice_product(sh, jb.P[1], jb.P[2], k, w, U, false);
            if (sh->abort) break;
            const double fs = bad ? NAN : ldexp(1.0, 2 * el);
            auto prow = [&](int q, int i) -> double { return fs * from_fixed(ld1(U + mat_at(k, i, q))); };
            if (lead) finish_column(s, a.pv, a.H, a.D, a.partial, prow, ls_smem, scratch, false, a.Sv);
            fence_proxy_async_smem();
            continue;
        }
        // (a submatrix that failed: NaN, not what the slot holds)
        const double fs = bad ? NAN : 0x1p-62;
        auto xrow = [&](int q, int i) -> double { return fs * static_cast<double>(ld1(X + mat_at(k, i, s.own + q))); };
        if (lead) finish_column(s, a.pv, a.H, a.D, a.partial, xrow, ls_smem, scratch);
        fence_proxy_async_smem();
        }
    }
    slices_end(sh);
    release_jobs(a.work_counter, a.ticket, reinterpret_cast<int*>(slot + 64));
}

// Setup of the non-orthogonal form for one (H, S) pair: from A_S (in Lc) and A_H (in Mc), both
// gathered without shift, L = A_S^-1/2 by the coupled iteration (into Lc) and M = L A_H L, exactly
// symmetric (into Mc), and the Gershgorin interval of M.
__global__ void __launch_bounds__(kSliceThreads, 1) k_nonorth_setup(const __grid_constant__ NonorthSetupArgs a) {
    __shared__ SliceShared shared;
    __shared__ SliceScalars ss;
    __shared__ SubDesc s;
    __shared__ SliceJob jb;
    __shared__ double scratch[64];
    SliceShared* const sh = &shared;
    slices_begin(sh, slice_stages(), a.status);
    uint8_t* slot = a.ws + static_cast<int64_t>(blockIdx.x / cluster_size()) * a.slot_bytes;
    for (int round = 0;; ++round) {
        const int job = claim_job(a.work_counter, &ss, &s, reinterpret_cast<int*>(slot + 64), round, a.n_subs, a.order, a.subs, a.Lc);
        if (job >= a.n_subs || sh->abort) break;
        if (threadIdx.x == 0) {
            slice_job(jb, slot + kSlotHead, s.n, a.kmax, a.mats);
            jb.scratch = reinterpret_cast<float*>(slot);
            jb.sums = reinterpret_cast<unsigned long long*>(slot + a.slot_bytes - sums_bytes(a.kmax));
        }
        __syncthreads();
        set_accumulation(sh, 7, kSliceK / 16);
        bool conv = false, bad = false;
        int ez = 0;
        const int done = coupled_steps(sh, jb, a.Lc + s.t_off, s.ld, a.bound_s[s.col], a.max_iter, static_cast<float>(a.tau), false, true, ez, &ss, conv, bad);
        if (sh->abort) break;
        if (done < 0) {
            if (threadIdx.x == 0 && cluster_rank() == 0) list_graded(a.graded, s.col);
            continue;
        }
        if (threadIdx.x == 0 && cluster_rank() == 0) {
            a.root_graded[s.col] = ss.graded;
            a.iters[s.col] = done;
            if (bad) atomicCAS(a.status, kOk, kErrNonfinite);
            else if (!conv) atomicCAS(a.status, kOk, kErrNoconv);
        }
        if (bad) {  // no L: the bracket is not used, the status tells
            if (threadIdx.x == 0 && cluster_rank() == 0) a.lohi[2 * s.col] = a.lohi[2 * s.col + 1] = 0.0;
            continue;
        }
        // A_H 2^-eh with rows of at most 1; Q = A_H L, then M = L Q = L A_H L: the right factor's digits
        // are those of Q^T, whose rows are Q's columns
        const int eh = load_fixed(a.Mc + s.t_off, s.ld, 0.0, 0.0, jb, jb.M[0], jb.P[0], kSource, sh, &ss);
        if (ss.bad) {
            if (threadIdx.x == 0 && cluster_rank() == 0) {
                atomicCAS(a.status, kOk, kErrNonfinite);
                a.lohi[2 * s.col] = a.lohi[2 * s.col + 1] = 0.0;
            }
            continue;
        }
        if (ss.graded) {
            if (threadIdx.x == 0 && cluster_rank() == 0) list_graded(a.graded, s.col);
            continue;
        }
        set_accumulation(sh, 8, 160 / 16);
        slice_product(sh, jb.P[0], jb.P[1], jb.k, jb.k, jb.M[2], false);
        if (sh->abort) break;
        // columns of A_H L may be longer than 1 (the 2-norm of A_H exceeds that of its rows)
        const float cn = column_norm2(jb, jb.M[2], sh);
        const int ep = cn > 1.0f ? static_cast<int>(ceilf(0.5f * log2f(cn * 1.001f))) : 0;
        pass_transposed(jb.M[2], nullptr, 0, jb.k, jb.P[2], jb.k, jb.k, ep);
        slice_product(sh, jb.P[1], jb.P[2], jb.k, jb.k, jb.M[2], true);
        if (sh->abort) break;
        const double b = a.bound_s[s.col];  // A_S^-1/2 = Z / sqrt(b)
        store_scaled(jb.M[1], jb.k, ldexp(1.0 / sqrt(b), ez - 62), a.Lc + s.t_off, s.n, s.ld);
        store_scaled(jb.M[2], jb.k, ldexp(1.0 / b, 2 * ez + eh + ep - 62), a.Mc + s.t_off, s.n, s.ld);
        if (cluster_size() > 1) phase_sync();
        else __syncthreads();
        if (cluster_rank() != 0) continue;
        const double2 g = gershgorin_interval(a.Mc + s.t_off, s.n, s.ld, scratch);
        if (threadIdx.x == 0) {
            a.lohi[2 * s.col] = g.x;
            a.lohi[2 * s.col + 1] = g.y;
        }
    }
    slices_end(sh);
    release_jobs(a.work_counter, a.ticket, reinterpret_cast<int*>(slot + 64));
}

size_t fp64_slot_bytes(int max_n, int mats, int planes) {
    const int64_t k = (static_cast<int64_t>(max_n) + 31) & ~int64_t(31);
    return static_cast<size_t>(kSlotHead + mats * k * k * 8 + planes * slice_bytes(k) + sums_bytes(k));
}

// n_clusters clusters of `size` CTAs.
template <class... P, class... A>
static cudaError_t launch_clusters(void (*kernel)(P...), int n_clusters, int size, cudaStream_t st, const A&... args) {
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(kSliceSmem));
    if (e != cudaSuccess) return e;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = static_cast<unsigned>(size);
    attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(static_cast<unsigned>(n_clusters * size));
    cfg.blockDim = dim3(kSliceThreads);
    cfg.dynamicSmemBytes = kSliceSmem;
    cfg.stream = st;
    cfg.attrs = &attr;
    cfg.numAttrs = size > 1 ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

// CTAs that a submatrix of n rows has work for: at most one per tile of 32 columns of its symmetric products
// (a power of two up to 8).
static int cluster_for(int n) {
    const int k = (n + 31) & ~31;
    int tiles = 0;
    for (int r = 0; r < k; r += 128) tiles += (k - r) / 32;
    return tiles >= 8 ? 8 : tiles >= 4 ? 4 : tiles >= 2 ? 2 : 1;
}

// CTAs per submatrix: as many as find room at once for all n_subs of them, at most cluster_for(max_n); one each where
// not even pairs do.  room[i]: clusters of 2^i CTAs the device holds at once (device_clusters; 76 pairs here, about 36
// fours and 18 eights).  Density builds of n_subs submatrices of n = 120 .. 204 with one CTA, two and four each, us:
//   8: 985 / 614 / 447 (eight: 331)   32: 1002 / 622 / 456    37: 1008 / 620 / 485    64: 1014 / 637 / 790
//   75: 1027 / 652 / 960    96: 1046 / 961 / 1140    128: 1082 / 1092 / 1515    256: 2042 / 2034 / 2928    304: 2166 / 2327 / 3402
// At the lines the larger cluster still wins where all fit, and four lose as soon as they do not.  Pairs past 76 gain
// where one CTA each leaves a short last wave (152: 1958 / 1315, 200: 2007 / 1588) and lose from about 300 on;
// telling those apart needs the submatrices' sizes, which the rule does not look at.
template <class K, class A>
static cudaError_t launch_form(K kernel, const A& a, int slots, int max_n, const int* room, cudaStream_t st) {
    int size = cluster_for(max_n), i = size == 8 ? 3 : size == 4 ? 2 : size == 2 ? 1 : 0;
    while (i > 0 && a.n_subs > room[i]) --i;
    return launch_clusters(kernel, slots, 1 << i, st, a);
}

// room[i]: how many clusters of 2^i CTAs of the kernel the device holds at once, i = 0 .. 3.
template <class K>
static cudaError_t kernel_clusters(K kernel, int* room) {
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(kSliceSmem));
    for (int i = 0; i < 4 && e == cudaSuccess; ++i) {
        cudaLaunchAttribute attr;
        attr.id = cudaLaunchAttributeClusterDimension;
        attr.val.clusterDim.x = 1u << i;
        attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(1u << i);
        cfg.blockDim = dim3(kSliceThreads);
        cfg.dynamicSmemBytes = kSliceSmem;
        cfg.attrs = &attr;
        cfg.numAttrs = 1;
        e = cudaOccupancyMaxActiveClusters(&room[i], kernel, &cfg);
    }
    return e;
}

cudaError_t device_clusters(int* room) { return kernel_clusters(k_ns_fp64<kFormSign>, room); }

cudaError_t launch_ns_fp64(const NsFp64Args& a, int slots, int max_n, int max_nblk, const int* room, cudaStream_t st) {
    if (sizeof(int) * (static_cast<size_t>(max_nblk) + 1) > kSliceSmem - 1024) return cudaErrorInvalidValue;
    cudaError_t e;
    switch (a.function) {
        case kFnDensity: e = launch_form(k_ns_fp64<kFormSign>, a, slots, max_n, room, st); break;
        case kFnFermi: e = launch_form(k_ns_fp64<kFormFermi>, a, slots, max_n, room, st); break;
        default: e = launch_form(k_ns_fp64<kFormRoots>, a, slots, max_n, room, st);
    }
    if (e != cudaSuccess || a.finish_iters > 0) return e;
    return launch_ns_graded(a, slots, max_nblk, st);
}

cudaError_t launch_nonorth_setup(const NonorthSetupArgs& a, int slots, int max_n, const int* room, cudaStream_t st) {
    const cudaError_t e = launch_form(k_nonorth_setup, a, slots, max_n, room, st);
    return e != cudaSuccess ? e : launch_graded_setup(a, slots, st);
}

}  // namespace smx

// ---------------------------------------------------------------------------
// Allocation-free dense entry point (no counterpart in the paper).
//
// Some callers cannot allocate device memory when they need a result:
// plug-ins inside a host framework whose caching allocator already owns the
// whole device pool (a cudaMalloc of their own would fail or fragment it),
// and latency-critical loops that must never enter the driver's allocator
// (cudaMalloc/cudaFree can synchronise the device and take milliseconds).
// smx_dense_density_noalloc serves them: it takes caller-owned input and
// output buffers and keeps its Newton-Schulz work matrices in the fixed
// device array below, which every GPU that loads this library holds until the
// process exits.  The call itself synchronises its stream to return the status.
// ---------------------------------------------------------------------------

#include <cmath>
#include <mutex>

#include "smx.h"

namespace smx {

namespace {
constexpr int kNoAllocMaxN = 256;                          // largest n accepted
constexpr int64_t kNoAllocMat = int64_t(kNoAllocMaxN) * kNoAllocMaxN;
constexpr int kNoAllocMaxDevices = 64;
}  // namespace

// The slot of one CTA (two matrices of 64-bit integers and the digits of two operands) for n = 256,
// followed by a small header: [0] status, [1] iterations, [2] rows of very different size (for k_dense_graded, with a bound
// of their length at [4]).  About 2.8 MiB.
constexpr int64_t kNoAllocBytes = kSlotHead + 2 * kNoAllocMat * 8 + 2 * slice_bytes(kNoAllocMaxN);
static __device__ __align__(256) uint8_t g_noalloc_scratch[kNoAllocBytes + 32];

// One cluster: D = 1/2 (I - sign(H - mu I)) of a dense symmetric H by the iteration of k_ns_fp64.
__global__ void __launch_bounds__(kSliceThreads, 1) k_dense_density_noalloc(const double* __restrict__ H, int n, double mu,
                                                                            double* __restrict__ Dout, uint8_t* scratch,
                                                                            float tau, int max_iter) {
    __shared__ SliceShared shared;
    __shared__ SliceScalars ss;
    __shared__ SignBound sb;
    int* hdr = reinterpret_cast<int*>(scratch + kNoAllocBytes);
    if (threadIdx.x == 0 && cluster_rank() == 0) hdr[0] = kOk, hdr[2] = 0;
    SliceShared* const sh = &shared;
    slices_begin(sh, slice_stages(), hdr);
    // every call overwrites the work matrices in full; nothing is carried over
    __shared__ SliceJob jb;
    if (threadIdx.x == 0) {
        slice_job(jb, scratch + kSlotHead, n, kNoAllocMaxN, 2);
        jb.scratch = reinterpret_cast<float*>(scratch);
    }
    __syncthreads();
    const int e = load_fixed(H, n, mu, 0.0, jb, jb.M[0], jb.P[0], kSource, sh, &ss);
    bool conv = false, bad = ss.bad != 0;
    int done = 0;
    const bool graded = !bad && ss.graded;
    if (!bad && !graded) done = sign_steps(sh, jb, e, max_iter, tau, 0, nullptr, &sb, &ss, conv, bad);
    const bool aborted = *static_cast<volatile int*>(&sh->abort) != 0;
    if (!aborted && !graded) {
        const int64_t* X = jb.M[0];
        for (int r = cluster_rank() * kSliceWarps + (threadIdx.x >> 5); r < n; r += cluster_size() * kSliceWarps)
            for (int c = threadIdx.x & 31; c < n; c += 32) {  // 1/2 (I - X) in units of 2^-63: up to 2^63
                const int64_t x = ld1(X + mat_at(jb.k, c, r)), one = r == c ? kFixedOne : 0;
                if (bad) {  // (no iterate: the array holds the last call's)
                    Dout[static_cast<int64_t>(r) * n + c] = NAN;
                    continue;
                }
                const bool negative = x > one;
                const uint64_t d = static_cast<uint64_t>(one) - static_cast<uint64_t>(x);
                Dout[static_cast<int64_t>(r) * n + c] = fixed_to_double(negative ? 0 - d : d, negative, -63);
            }
    }
    slices_end(sh);
    if (threadIdx.x == 0 && cluster_rank() == 0) {
        if (graded) {
            hdr[2] = 1;
            *reinterpret_cast<double*>(hdr + 4) = ldexp(1.0, e);
        }
        if (!aborted && !graded) atomicCAS(hdr, kOk, bad ? kErrNonfinite : (conv ? kOk : kErrNoconv));
        hdr[1] = done;
    }
}

}  // namespace smx

namespace {
std::mutex g_noalloc_mutex;
// per device: the array's device address and the context it was looked up in
uint8_t* g_noalloc_ptr[smx::kNoAllocMaxDevices] = {};
CUcontext g_noalloc_ctx[smx::kNoAllocMaxDevices] = {};
// the CTAs of the largest cluster it has room for there
int g_noalloc_cluster[smx::kNoAllocMaxDevices] = {};

// The current driver context, through the runtime's driver entry point (no link to libcuda).
CUcontext current_context() {
    using Fn = CUresult (*)(CUcontext*);
    static Fn fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuCtxGetCurrent", &p, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<Fn>(p);
    });
    CUcontext c = nullptr;
    if (fn) fn(&c);
    return c;
}
}  // namespace

extern "C" smx_status smx_dense_density_noalloc(const double* h_dev, int32_t n, double mu, double* d_dev,
                                                void* cuda_stream) {
    if (!h_dev || !d_dev || n < 1 || n > smx::kNoAllocMaxN || !std::isfinite(mu)) return SMX_ERR_ARG;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return SMX_ERR_CUDA;
    if (dev < 0 || dev >= smx::kNoAllocMaxDevices) return SMX_ERR_UNSUPPORTED;
    uint8_t* scratch = nullptr;
    int largest = 1;
    {
        // set-up once per device, with that device current: the host-side name
        // of a __device__ array is not a device address, so look the address up.
        // A device reset (cudaDeviceReset) replaces the context and reloads the
        // module, so the lookup is repeated when the current context changed.
        std::lock_guard<std::mutex> lock(g_noalloc_mutex);
        const CUcontext cur = current_context();
        if (!g_noalloc_ptr[dev] || g_noalloc_ctx[dev] != cur) {
            void* p = nullptr;
            if (cudaGetSymbolAddress(&p, smx::g_noalloc_scratch) != cudaSuccess || !p) return SMX_ERR_CUDA;
            int room[4] = {0, 0, 0, 0};
            if (smx::kernel_clusters(smx::k_dense_density_noalloc, room) != cudaSuccess) return SMX_ERR_CUDA;
            g_noalloc_cluster[dev] = room[3] > 0 ? 8 : room[2] > 0 ? 4 : room[1] > 0 ? 2 : 1;
            g_noalloc_ptr[dev] = static_cast<uint8_t*>(p);
            g_noalloc_ctx[dev] = cur;
        }
        scratch = g_noalloc_ptr[dev];
        largest = g_noalloc_cluster[dev];
    }
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    const int size = smx::cluster_for(n) < largest ? smx::cluster_for(n) : largest;
    if (smx::launch_clusters(smx::k_dense_density_noalloc, 1, size, st, h_dev, static_cast<int>(n), mu, d_dev, scratch, 1e-7f, 100) != cudaSuccess)
        return SMX_ERR_CUDA;
    int* const head = reinterpret_cast<int*>(scratch + smx::kNoAllocBytes);
    if (smx::launch_dense_graded(h_dev, static_cast<int>(n), mu, d_dev, scratch, 1e-7, 100, head + 2, reinterpret_cast<double*>(head + 4), head, st) !=
        cudaSuccess)
        return SMX_ERR_CUDA;
    int hdr[2] = {0, 0};
    if (cudaMemcpyAsync(hdr, scratch + smx::kNoAllocBytes, sizeof(hdr), cudaMemcpyDeviceToHost, st) != cudaSuccess)
        return SMX_ERR_CUDA;
    if (cudaStreamSynchronize(st) != cudaSuccess) return SMX_ERR_CUDA;
    return static_cast<smx_status>(hdr[0]);
}
