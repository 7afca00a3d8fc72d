// 64-bit symmetric-matrix products on the tcgen05 tensor cores by error-free slices (the Ozaki
// splitting of Ozaki, Ogita, Oishi and Rump, Numer. Algorithms 59, 2012, with FP16 slices and
// FP32 accumulation as in Mukunoki et al., ISC 2020).
//
// A cluster of CTAs may share the work of a submatrix: the tiles of a product and the units of an
// elementwise pass go round the CTAs; whatever is decided from a reduction is decided alike by each.
//
// Numbers.  A matrix is held in fixed point: 64-bit integers in units of 2^-62.  An operand of a
// product is cut into seven 8-bit digits,
//     x = sum_{i=1..7} d_i 2^(-8 i),   |d_1| <= 256 (1 + a little), |d_i| <= 128,
// i.e. rounded to 2^-56.  The digits are small integers, exact in FP16; a tensor-core product of
// two digit matrices sums integers, and every sum below stays within 2^24, so the FP32
// accumulators in tensor memory hold it exactly.  The pairs (i, j) of one weight g = i + j share
// an accumulator; g = 2 .. 8 (28 pairs) are kept.  The epilogue adds the seven accumulators as
// integers with their weights, so the only errors of a product are the 2^-57 rounding of the
// operands and the dropped weights g >= 9: about 3.4e-17 sqrt(K / 158) per entry, below the
// rounding of a chain of K FP64 fused multiply-adds on entries of order 0.1 .. 1.  (In units of the matrix's
// longest row: rows much shorter than that would lose digits, and are not multiplied here; kGraded.)
//
// Exactness.  The rows of both operands have 2-norms of at most 1.05 (the callers scale by a
// power of two where it takes one).  So |sum_k d_1 d_j| <= 256 * 1.05 * 128 sqrt(K) for j > 1, and
// the largest accumulator, g = 8, holds at most 2 * 1.05 * 2^15 sqrt(K) + 5 * 2^14 K < 2^24 for
// K <= 192 (kSliceK): longer contractions are summed in parts of 192 (in parts of 160 where one
// operand's rows may reach a norm of 2).
//
// Why: GB300's FP64 units take about 16 cycles per warp instruction and SM (1.2 TFLOP/s for the
// GPU); 28 FP16 products on the tensor cores (2 PFLOP/s) are some 50 times faster.
//
// Layout.  The digits of an operand live in global memory (L2) as seven planes in the canonical
// K-major layout with the 32-byte swizzle: for each block of 128 rows, for each group of 16 columns k
// (a chunk), for each plane, the block's rows of 32 bytes one after the other.  Both factors of C =
// A B^T are read that way (every right factor here is symmetric, or is kept transposed): the left
// factor's chunk of a tile is one bulk copy (cp.async.bulk), the right factor's one per plane.  The B
// planes of a chunk lie one after the other in shared memory, so that one instruction multiplies
// A's plane i by B's planes 1 .. 8 - i at once (N = 64 (8 - i), in one or two parts): their products
// belong to the weights i + 1 .. 8, whose accumulators are neighbouring columns of tensor memory.
// A matrix of 64-bit integers with k rows is stored by pairs of columns: entry (r, c) at
// ((c >> 1) k + r) 2 + (c & 1), so that the lanes of a warp, which hold consecutive rows, read and
// write 16 bytes each side by side.
#pragma once

#include "smx_device.cuh"

namespace smx {

namespace {

constexpr int kSliceThreads = 512;  // 16 warps of up to 128 registers (spills would go to L2: shared memory leaves no L1)
constexpr int kSliceWarps = kSliceThreads / 32;
constexpr int kSliceAdders = 14;    // of these read the accumulators; warp 0 copies, warp 1 issues the products
constexpr int kSlicePlanes = 7;
constexpr int kSliceK = 192;        // K of one exact accumulation (see above)
constexpr int kSliceTile = 64;      // columns of a tile: seven (eight) accumulators of 64 columns
constexpr int kSliceStages = 5;     // chunks of 16 K in shared memory
constexpr uint32_t kSliceABytes = kSlicePlanes * 128 * 32;
constexpr uint32_t kSliceStageBytes = kSliceABytes + kSlicePlanes * kSliceTile * 32;
constexpr size_t kSliceSmem = 1024 + static_cast<size_t>(kSliceStages) * kSliceStageBytes;

// Bytes of the planes of a k x k operand (k a multiple of 32).
__host__ __device__ constexpr int64_t slice_bytes(int64_t k) { return kSlicePlanes * k * k * 2; }

// The CTA's state in shared memory (kept out of registers: they would be spilled around the products).
struct SliceShared {
    uint64_t full[kSliceStages], empty[kSliceStages], tfull, tempty, drain;
    uint8_t* smem;   // 1024-byte aligned stages
    int* status;
    uint32_t tmem;
    int abort;
    int gave_up[2];  // abort as the readers of an accumulation all see it (by its number modulo 2)
    int kpart;       // chunks of one exact accumulation (fewer than kSliceK / 16 where an operand's rows are longer)
    int tile;        // columns of a tile: kSliceTile, or half of it to have tiles for all CTAs of a larger cluster
    int weights;     // 7: the pairs of weights 2 .. 8; 8: of weight 9 too (kpart at most 10)
    // positions of the roles in the pipelines, continuous over the products of a CTA: chunks copied,
    // chunks multiplied, accumulations begun, accumulations read (each written by one role)
    uint32_t copied, multiplied, begun, read;
    uint4 list[24];  // the products of a chunk: A and B offsets, first column, instruction descriptor, opens its columns
    float red[2 * kSliceWarps];
};

// 16-byte aligned bulk copy global -> shared, counted on an mbarrier.
__device__ __forceinline__ void bulk_load(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(smem_u32(dst)),
                 "l"(src), "r"(bytes), "r"(smem_u32(bar))
                 : "memory");
}

// Shared-memory descriptor of a K-major operand of 16 K values (32-byte rows, 32-byte swizzle).
__device__ __forceinline__ uint64_t sdesc_sw32(uint32_t saddr) {
    uint64_t d = 0;
    d |= static_cast<uint64_t>((saddr & 0x3FFFFu) >> 4);
    d |= static_cast<uint64_t>(1) << 16;          // leading byte offset (unused for swizzled K-major)
    d |= static_cast<uint64_t>(256 >> 4) << 32;   // stride byte offset: eight rows
    d |= static_cast<uint64_t>(1) << 46;          // descriptor version
    d |= static_cast<uint64_t>(6) << 61;          // 32-byte swizzle
    return d;
}

// 4 consecutive 32-bit TMEM columns of this thread's lane; the registers are valid only after
// tmem_wait4x4, which names them so that nothing uses (or moves) them before.
__device__ __forceinline__ void tmem_ld4(uint32_t taddr, uint32_t (&r)[4]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(taddr));
}
__device__ __forceinline__ void tmem_wait4x4(uint32_t (&a)[4], uint32_t (&b)[4], uint32_t (&c)[4], uint32_t (&d)[4]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(a[0]), "+r"(a[1]), "+r"(a[2]), "+r"(a[3]), "+r"(b[0]), "+r"(b[1]), "+r"(b[2]), "+r"(b[3]), "+r"(c[0]),
                   "+r"(c[1]), "+r"(c[2]), "+r"(c[3]), "+r"(d[0]), "+r"(d[1]), "+r"(d[2]), "+r"(d[3])
                 :
                 : "memory");
}
// An accumulator (an integer of at most 2^24 in magnitude) as an integer; acc_small: of at most 2^22
// (weights 2 .. 4: 2.1 * 2^15 sqrt(K) + 2^14 K < 2^22 for K <= 192), by an addition instead of the
// conversion, which has a quarter of the rate.
__device__ __forceinline__ int acc_int(uint32_t v) { return __float2int_rn(__uint_as_float(v)); }
__device__ __forceinline__ int acc_small(uint32_t v) {
    return __float_as_int(__fadd_rn(__uint_as_float(v), 12582912.0f)) - 0x4B400000;  // 1.5 * 2^23
}
// A quarter of an accumulator, rounded; and acc_int in two steps of that kind (a multiple of four and a
// remainder of -2 .. 2), so that not every accumulator waits for the conversion unit.
__device__ __forceinline__ int acc_quarter(uint32_t v) {
    return __float_as_int(__fadd_rn(__uint_as_float(v), 50331648.0f)) - 0x4C400000;  // 1.5 * 2^25
}
__device__ __forceinline__ int acc_steps(uint32_t v) {
    const float x = __uint_as_float(v), t = __fadd_rn(x, 50331648.0f);
    return 4 * (__float_as_int(t) - 0x4C400000) + acc_small(__float_as_uint(__fsub_rn(x, __fsub_rn(t, 50331648.0f))));
}

// Entries (r, c .. c + 7) of a matrix with k rows (c even).
__device__ __forceinline__ int64_t mat_at(int k, int r, int c) {
    return ((static_cast<int64_t>(c >> 1) * k + r) << 1) + (c & 1);
}
__device__ __forceinline__ void ld8(const int64_t* m, int k, int r, int c, int64_t (&v)[8]) {
    const longlong2* p = reinterpret_cast<const longlong2*>(m) + static_cast<int64_t>(c >> 1) * k + r;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const longlong2 x = __ldcg(p + static_cast<int64_t>(i) * k);
        v[2 * i] = x.x;
        v[2 * i + 1] = x.y;
    }
}
__device__ __forceinline__ void st8(int64_t* m, int k, int r, int c, const int64_t (&v)[8]) {
    longlong2* p = reinterpret_cast<longlong2*>(m) + static_cast<int64_t>(c >> 1) * k + r;
#pragma unroll
    for (int i = 0; i < 4; ++i) p[static_cast<int64_t>(i) * k] = make_longlong2(v[2 * i], v[2 * i + 1]);
}

// Sets up the barriers and all of tensor memory; all threads call it.
__device__ void slices_begin(SliceShared* sh, uint8_t* smem, int* status) {
    if (threadIdx.x == 0) {
        sh->smem = smem;
        sh->status = status;
        sh->kpart = kSliceK / 16;
        sh->weights = 7;
        sh->tile = cluster_size() >= 4 ? kSliceTile / 2 : kSliceTile;
        sh->copied = sh->multiplied = sh->begun = sh->read = 0;
        for (int s = 0; s < kSliceStages; ++s) {
            mbar_init(&sh->full[s], 1);
            mbar_init(&sh->empty[s], 1);
        }
        mbar_init(&sh->tfull, 1);
        mbar_init(&sh->tempty, kSliceAdders);
        mbar_init(&sh->drain, 1);
        sh->abort = 0;
        fence_barrier_init();
    }
    if (threadIdx.x >= 32 && threadIdx.x < 64) tmem_alloc(&sh->tmem, 512);
    __syncthreads();
    tc_fence_after();
}

// Ends the CTA's use of tensor memory; after a timeout the copies and products in flight are
// waited for (bounded) first.  All threads call it.
__device__ void slices_end(SliceShared* sh) {
    __syncthreads();
    volatile int* ab = &sh->abort;
    auto wait_some = [](uint64_t* bar, uint32_t parity) {
        for (uint32_t i = 0; i < (1u << 20); ++i)
            if (mbar_try_wait(bar, parity)) return;
    };
    if (*ab && threadIdx.x == 0)
        for (uint32_t it = sh->multiplied; it < sh->copied; ++it) wait_some(&sh->full[it % kSliceStages], (it / kSliceStages) & 1);
    if (*ab && threadIdx.x >= 32 && threadIdx.x < 64 && elect_one()) {  // the lane that issued the products
        tc_commit(&sh->drain);
        wait_some(&sh->drain, 0);
    }
    __syncthreads();
    if (threadIdx.x >= 32 && threadIdx.x < 64) {
        tc_fence_after();
        tmem_dealloc(sh->tmem, 512);
    }
}

// C = A B^T as 64-bit integers in units of 2^-62: A is k x k in planes pa (k a multiple of 32), B has
// kb rows (a multiple of 16) of k in planes pb; C has k rows and kb columns.  sym: the product is
// symmetric (kb = k): only the tiles on and right of the diagonal 128 x 128 blocks are multiplied, the
// upper triangle is kept and mirrored, so that C is exactly symmetric.  All threads call it; the
// planes were written before a proxy fence and a barrier.  Ends with a barrier.
//
// A tile has 128 rows and 64 columns.  Per chunk of 16 K: 28 digit products of 128 x 64 x 16 in 10
// instructions, 910 cycles (2 accumulator columns a cycle, the tensor cores' rate) at 46 bytes of
// planes per cycle.  Warp 0 copies up to five chunks ahead, one lane of warp 1 issues the products;
// (n = 150, k = 160: about 64,000 cycles a product, 29,000 of them the tensor cores' own and some 40,000 the
// operands' shared-memory reads; the reading of the last tile is not hidden)
// the other 14 read a finished tile's accumulators (a warp its quadrant's 32 rows, the quadrant's warps
// four columns each in turn), then free them for the next tile before they write C.
__device__ __noinline__ void slice_product(SliceShared* sh, const uint8_t* __restrict__ pa, const uint8_t* __restrict__ pb, int k,
                                           int kb, int64_t* __restrict__ C, bool sym) {
    uint8_t* smem = sh->smem;
    int* const status = sh->status;
    volatile int* ab = &sh->abort;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int mtiles = (k + 127) >> 7, chunks = k >> 4;
    const int kpart = sh->kpart, weights = sh->weights, tile = sh->tile;
    const int ranks = cluster_size(), rank = cluster_rank();
    const int parts = (chunks + kpart - 1) / kpart;
    const uint32_t tmem = sh->tmem;
    if (warp == 0) {
        if (elect_one()) {
            const int64_t blk = static_cast<int64_t>(k) * 128 * kSlicePlanes * 2;  // bytes of a block of 128 rows
            uint32_t it = sh->copied;
            bool ok = true;
            int turn = 0;
            for (int mt = 0; mt < mtiles && ok; ++mt)
                for (int c0 = sym ? 128 * mt : 0; c0 < kb && ok; c0 += tile) {
                    if (turn++ % ranks != rank) continue;
                    const uint32_t ra = static_cast<uint32_t>(min(128, k - 128 * mt)) * 32, w = static_cast<uint32_t>(min(tile, kb - c0)) * 32;
                    const uint32_t rb = static_cast<uint32_t>(min(128, kb - (c0 & ~127))) * 32;
                    const uint8_t* a = pa + mt * blk;
                    const uint8_t* b = pb + (c0 >> 7) * blk + (c0 & 127) * 32;
                    for (int kc = 0; kc < chunks; ++kc, ++it) {
                        const int stage = it % kSliceStages;
                        if (it >= kSliceStages && !mbar_wait(&sh->empty[stage], (it / kSliceStages - 1) & 1, ab, status)) {
                            ok = false;
                            break;
                        }
                        mbar_arrive_expect_tx(&sh->full[stage], kSlicePlanes * (ra + w));
                        uint8_t* s = smem + static_cast<uint32_t>(stage) * kSliceStageBytes;
                        bulk_load(s, a, kSlicePlanes * ra, &sh->full[stage]);
#pragma unroll
                        for (int p = 0; p < kSlicePlanes; ++p) bulk_load(s + kSliceABytes + p * w, b + p * rb, w, &sh->full[stage]);
                        a += kSlicePlanes * ra;
                        b += kSlicePlanes * rb;
                    }
                }
            sh->copied = it;
        }
        __syncwarp();
    } else if (warp == 1) {
        bool alive = true;
        int turn = 0;
        for (int mt = 0; mt < mtiles && alive; ++mt)
            for (int c0 = sym ? 128 * mt : 0; c0 < kb && alive; c0 += tile) {
                if (turn++ % ranks != rank) continue;
                // The products of one chunk, the same for every chunk of the tile, listed once (a lane per
                // product): formed in the issuing loop, their descriptors would take longer than the products.
                // A's plane i (from 1) takes B's planes 1 .. j1 = min(7, weights + 1 - i), in one or two
                // instructions of N <= 256.  In the first chunk plane 1 opens the accumulators; that of weight
                // 9 is opened by planes 2 and 7, on their own.
                const int w = min(tile, kb - c0);
                int count;
                {
                    const uint32_t ra = static_cast<uint32_t>(min(128, k - 128 * mt)) * 32;
                    const int i = 1 + lane / 3, piece = lane - 3 * (i - 1);
                    const bool open9 = i == 2 && weights == 8;
                    const int total = w * (min(kSlicePlanes, weights + 1 - i) - (open9 ? 1 : 0)), step = total > 256 ? total >> 1 : total;
                    const int at = piece == 2 ? total : piece * step;  // columns from plane 1's on
                    const int n = piece == 2 ? (open9 ? w : 0) : at < total ? step : 0;
                    const bool valid = i <= kSlicePlanes && n > 0;
                    const uint32_t mask = __ballot_sync(0xffffffffu, valid);
                    count = __popc(mask);
                    if (valid)
                        sh->list[__popc(mask & ((1u << lane) - 1u))] =
                            make_uint4(((i - 1) * ra) >> 4, (kSliceABytes + at * 32) >> 4, tmem + (i - 1) * w + at,
                                       idesc_f16(128, n, 0) | (i == 1 || piece == 2 ? 1u : 0u));
                    __syncwarp();
                }
                int ok = 1;
                if (elect_one()) {
                    // the queue of the tensor cores holds only a few products: little between two chunks
                    const uint64_t desc0 = sdesc_sw32(0) + (smem_u32(smem) >> 4);
                    const uint32_t it0 = sh->multiplied;
                    uint32_t stage = it0 % kSliceStages, phase = (it0 / kSliceStages) & 1, use = sh->begun;
                    uint64_t base = desc0 + stage * (kSliceStageBytes >> 4);
                    int kc = 0;
                    while (kc < chunks && ok) {
                        const int end = min(chunks, kc + kpart);  // of this accumulation
                        if (use++ > 0) ok = mbar_wait(&sh->tempty, (use - 2) & 1, ab, status);
                        tc_fence_after();
                        uint32_t keep = 0;
                        for (; kc < end; ++kc) {
                            if (!mbar_try_wait(&sh->full[stage], phase) && !mbar_wait(&sh->full[stage], phase, ab, status)) {
                                ok = 0;
                                break;
                            }
#pragma unroll 4
                            for (int e = 0; e < count; ++e) {
                                const uint4 p = sh->list[e];
                                tc_mma_f16(p.z, base + p.x, base + p.y, p.w & ~1u, keep | (~p.w & 1u));
                            }
                            tc_commit(&sh->empty[stage]);
                            keep = 1;
                            base += kSliceStageBytes >> 4;
                            if (++stage == kSliceStages) {
                                stage = 0;
                                phase ^= 1;
                                base = desc0;
                            }
                        }
                        if (ok) tc_commit(&sh->tfull);
                    }
                    sh->multiplied = it0 + kc;
                    sh->begun = use;
                }
                __syncwarp();
                alive = *ab == 0;
            }
    } else {
        const int q = warp & 3;  // lanes 32 q .. of tensor memory
        const int idx = q < 2 ? (warp >> 2) - 1 : warp >> 2, cnt = q < 2 ? 3 : 4;  // among the quadrant's warps
        constexpr int kTurns = (kSliceTile / 4 + 2) / 3;
        uint32_t use = sh->read;
        bool alive = true;
        int turn = 0;
        for (int mt = 0; mt < mtiles && alive; ++mt)
            for (int c0 = sym ? 128 * mt : 0; c0 < kb && alive; c0 += tile) {
                if (turn++ % ranks != rank) continue;
                const int w = min(tile, kb - c0);
                int64_t sum[kTurns][4];
                for (int p = 0; p < parts; ++p) {
                    // one lane polls; the other warps wait at a barrier without touching shared memory, whose
                    // bandwidth the products need.  That lane's one look at the abort flag decides for all: each
                    // looking for itself, a flag raised in between would leave some of them at this barrier for good.
                    if (warp == 2 && lane == 0) {
                        mbar_wait(&sh->tfull, use & 1, ab, status);
                        sh->gave_up[use & 1] = *ab;
                    }
                    asm volatile("bar.sync 1, 448;" ::: "memory");
                    alive = !sh->gave_up[use & 1];
                    ++use;
                    if (!alive) break;
                    tc_fence_after();
#pragma unroll
                    for (int h = 0; h < kTurns; ++h) {
                        const int c = 4 * (idx + cnt * h);
                        if (c >= w) break;
                        // weights 2 .. 9 in units of 2^-62: 2^46, 2^38, 2^30, 2^22, 2^14, 2^6, 2^-2, 2^-10
                        const uint32_t col = tmem + (static_cast<uint32_t>(q * 32) << 16) + c;
                        uint32_t v0[4], v1[4], v2[4], v3[4];
                        tmem_ld4(col, v0);
                        tmem_ld4(col + w, v1);
                        tmem_ld4(col + 2 * w, v2);
                        tmem_ld4(col + 3 * w, v3);
                        tmem_wait4x4(v0, v1, v2, v3);
                        int64_t s[4];
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            s[i] = static_cast<int64_t>(acc_int(v3[i])) * (1 << 22) + static_cast<int64_t>(acc_small(v2[i])) * (1 << 30);
                            const int hi = acc_small(v1[i]) * 64 + acc_small(v0[i]) * (1 << 14);
                            s[i] += static_cast<int64_t>(static_cast<uint64_t>(static_cast<uint32_t>(hi)) << 32);
                        }
                        tmem_ld4(col + 4 * w, v0);
                        tmem_ld4(col + 5 * w, v1);
                        tmem_ld4(col + 6 * w, v2);
                        if (weights == 8) tmem_ld4(col + 7 * w, v3);
                        tmem_wait4x4(v0, v1, v2, v3);
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            int tail = acc_quarter(v2[i]);
                            if (weights == 8) tail = ((acc_int(v2[i]) << 4) + ((acc_int(v3[i]) + 8) >> 4) + 32) >> 6;
                            s[i] += static_cast<int64_t>(acc_int(v0[i])) * (1 << 14) + static_cast<int64_t>(acc_steps(v1[i])) * 64 + tail;
                            sum[h][i] = p == 0 ? s[i] : sum[h][i] + s[i];
                        }
                    }
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&sh->tempty);
                }
                const int r0 = 128 * mt + 32 * q, row = r0 + lane;
                if (alive && r0 < k) {  // k is a multiple of 32: uniform over the warp
#pragma unroll
                    for (int h = 0; h < kTurns; ++h) {
                        const int c = 4 * (idx + cnt * h), col = c0 + c;
                        if (c >= w) break;
                        if (!sym || col > r0 + 31) {
                            longlong2* d = reinterpret_cast<longlong2*>(C) + static_cast<int64_t>(col >> 1) * k + row;
                            d[0] = make_longlong2(sum[h][0], sum[h][1]);
                            d[k] = make_longlong2(sum[h][2], sum[h][3]);
                            if (sym) {
#pragma unroll
                                for (int i = 0; i < 4; ++i) C[mat_at(k, col + i, row)] = sum[h][i];
                            }
                        } else if (col + 3 >= r0) {  // the chunk of the warp's diagonal
#pragma unroll
                            for (int i = 0; i < 4; ++i)
                                if (col + i >= row) {
                                    C[mat_at(k, row, col + i)] = sum[h][i];
                                    C[mat_at(k, col + i, row)] = sum[h][i];
                                }
                        }
                    }
                }
            }
        if (warp == 2 && lane == 0) sh->read = use;  // (every reader took its copy before the last barrier)
    }
    phase_sync();
}

// Digits of eight neighbouring values of a row (units of 2^-62) to the seven planes, 16 bytes each.
// The offset makes every digit's byte non-negative (128 added to d_2 .. d_7, 512 to d_1); FP16
// 1024 + u is the bit pattern 0x6400 | u, from which the offset is subtracted exactly.
__device__ __forceinline__ void store_digits(const int64_t (&q)[8], uint8_t* dst, int64_t pstride) {
    uint32_t lo[8], hi[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const uint64_t t = static_cast<uint64_t>(((q[i] + 32) >> 6) + 0x0200808080808080ll);
        lo[i] = static_cast<uint32_t>(t);
        hi[i] = static_cast<uint32_t>(t >> 32);
    }
#pragma unroll
    for (int p = 0; p < kSlicePlanes; ++p) {
        uint32_t w[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            uint32_t x;
            if (p == 0) {
                x = __byte_perm(hi[2 * u], hi[2 * u + 1], 0x7632) | 0x64006400u;
            } else {
                const uint32_t a = p <= 2 ? hi[2 * u] : lo[2 * u], b = p <= 2 ? hi[2 * u + 1] : lo[2 * u + 1];
                constexpr uint32_t sel[7] = {0, 0x5511, 0x4400, 0x7733, 0x6622, 0x5511, 0x4400};
                x = (__byte_perm(a, b, sel[p]) & 0x00FF00FFu) | 0x64006400u;
            }
            const uint32_t off = p == 0 ? 0x66006600u : 0x64806480u;
            const __half2 d = __hsub2(*reinterpret_cast<const __half2*>(&x), *reinterpret_cast<const __half2*>(&off));
            w[u] = *reinterpret_cast<const uint32_t*>(&d);
        }
        *reinterpret_cast<uint4*>(dst + p * pstride) = make_uint4(w[0], w[1], w[2], w[3]);
    }
}

// An elementwise pass: f(r, c, v, q) turns the values v loaded by load(r, c, v) (eight from each of N
// matrices) into the values q = (r, c .. c + 7) of an operand of rows x k (zero past the matrix); their
// digits go to the planes (null: f alone).  Ends a phase.  Lane pairs take the two halves of a plane's
// 32-byte row, 16 rows a warp.
template <int N, class L, class F>
__device__ __forceinline__ void slice_pass(int rows, int k, uint8_t* planes, L load, F f) {
    const int first = cluster_rank() * kSliceThreads + threadIdx.x, step = cluster_size() * kSliceThreads;
    const int units = rows * (k >> 3), half = threadIdx.x & 1;
    int r = first >> 1, c = 8 * half;
    for (int u = first; u < units; u += step, r += step >> 1) {
        while (r >= rows) {
            r -= rows;
            c += 16;
        }
        int64_t v[N][8], q[8];
        load(r, c, v);
        f(r, c, v, q);
        if (planes) {
            const int rb = min(128, rows - (r & ~127));
            uint8_t* dst = planes + static_cast<int64_t>(r >> 7) * (static_cast<int64_t>(k) * 128 * kSlicePlanes * 2) +
                           (static_cast<int64_t>(c >> 4) * kSlicePlanes * rb + (r & 127)) * 32 + ((half ^ ((r >> 2) & 1)) << 4);
            store_digits(q, dst, static_cast<int64_t>(rb) * 32);
        }
    }
    phase_sync_copies();
}

// ---------------------------------------------------------------------------
// fixed-point arithmetic (units of 2^-62)
// ---------------------------------------------------------------------------

constexpr int64_t kFixedOne = int64_t(1) << 62;

// x f for a factor f < 16 in units of 2^-60 (fixed_factor), rounded (cut off four bits above the last,
// it was the largest error of the Fermi form).
__device__ __forceinline__ int64_t fixed_mul(int64_t x, uint64_t f60) {
    const uint64_t a = static_cast<uint64_t>(x < 0 ? -x : x), lo = a * f60;
    const uint64_t m = (__umul64hi(a, f60) << 4) + (lo >> 60) + ((lo >> 59) & 1u);
    return x < 0 ? -static_cast<int64_t>(m) : static_cast<int64_t>(m);
}
__device__ __forceinline__ uint64_t fixed_factor(double f) { return static_cast<uint64_t>(f * 0x1p60); }

// t f 2^-e in units of 2^-62, rounded; f in (1/2, 1] as a fraction of 2^64 (0: 1).  bad is set for a
// value that is not finite or not below 2.
__device__ __forceinline__ int64_t to_fixed(double t, int e, uint64_t f, bool& bad) {
    const uint64_t b = static_cast<uint64_t>(__double_as_longlong(t));
    const int ex = static_cast<int>((b >> 52) & 0x7ff);
    if (ex == 0) return 0;  // zero, subnormal
    uint64_t m = ((b & 0xfffffffffffffull) | 0x10000000000000ull) << 11;  // 2^63 .. 2^64: value m 2^(ex - 1086)
    if (f) m = __umul64hi(m, f);
    const int sh = 1024 + e - ex;  // right shift to units of 2^-62
    const uint64_t v = sh <= 0 ? m : sh <= 63 ? (m >> sh) + ((m >> (sh - 1)) & 1u) : 0u;
    if (ex == 0x7ff || sh < 0 || (v >> 63)) {
        bad = true;
        return 0;
    }
    return (b >> 63) ? -static_cast<int64_t>(v) : static_cast<int64_t>(v);
}
__device__ __forceinline__ double from_fixed(int64_t x) { return static_cast<double>(x) * 0x1p-62; }
// x as a float in units of 2^-38 to an error of 2^-38 or 2^-24 relative (for sums of squares)
__device__ __forceinline__ float fixed_float(int64_t x) {
    const bool big = static_cast<uint32_t>(static_cast<int>(x >> 55) + 1) > 1u;
    return static_cast<float>(static_cast<int>(big ? x >> 31 : x >> 24)) * (big ? 128.0f : 1.0f);
}

// +-a 2^ex as a double (ex >= -900), rounded to nearest, on the integer units.
__device__ __forceinline__ double fixed_to_double(uint64_t a, bool negative, int ex) {
    if (a == 0) return 0.0;
    const int lz = __clzll(static_cast<long long>(a));
    const uint64_t m = a << lz;  // leading bit at 63
    uint64_t r = m >> 11;
    const uint64_t rem = m & 0x7ffu;
    if (rem > 0x400u || (rem == 0x400u && (r & 1u))) ++r;  // a carry moves into the exponent: correct
    const uint64_t bits = r + (static_cast<uint64_t>(1023 + 63 - lz + ex - 1) << 52);
    return __longlong_as_double(static_cast<long long>(bits | (negative ? 0x8000000000000000ull : 0ull)));
}

// Sum / maximum over the CTA of one float per thread (every thread gets it; the same order always).
__device__ __forceinline__ float cta_sum(float v, SliceShared* sh) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) sh->red[threadIdx.x >> 5] = v;
    __syncthreads();
    float s = 0.0f;
    for (int w = 0; w < kSliceWarps; ++w) s += sh->red[w];
    return s;
}
// The sum over the cluster; scratch: one float per CTA in global memory.
__device__ __noinline__ float cluster_sum(float v, SliceShared* sh, float* scratch) {
    v = cta_sum(v, sh);
    const int ranks = cluster_size();
    if (ranks == 1) return v;
    if (threadIdx.x == 0) __stcg(scratch + cluster_rank(), v);
    phase_sync();
    float s = 0.0f;
    for (int r = 0; r < ranks; ++r) s += __ldcg(scratch + r);
    return s;
}
// The maximum over the cluster of one value per CTA (the same for its threads); scratch as above.
__device__ __forceinline__ uint32_t cluster_max(uint32_t v, uint32_t* scratch) {
    const int ranks = cluster_size();
    if (ranks == 1) return v;
    if (threadIdx.x == 0) __stcg(scratch + cluster_rank(), v);
    phase_sync();
    for (int r = 0; r < ranks; ++r) v = max(v, __ldcg(scratch + r));
    return v;
}
__device__ __forceinline__ float cta_max(float v, SliceShared* sh) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
    __syncthreads();
    if ((threadIdx.x & 31) == 0) sh->red[threadIdx.x >> 5] = v;
    __syncthreads();
    float s = 0.0f;
    for (int w = 0; w < kSliceWarps; ++w) s = fmaxf(s, sh->red[w]);
    return s;
}

}  // namespace

}  // namespace smx
