// cg_train.cu -- one training step of the learned initial guess in six
// launches, for batches up to kTrainRows rows.
//
// The products are those of tgemm_kernel (cg_mlp.cu): FP32 operands as TF32
// pairs hi + lo, three tcgen05.mma (kind::tf32) per eight K elements, FP32
// accumulation in tensor memory, the same K ranges for the weight gradients.
// There every block split its operands itself, from 4-byte copies, and a step
// was 19 launches (174 us for 1,024 rows).  Here whatever produces an operand
// -- the gather of the batch, an epilogue, the Adam step -- writes it once as
// an *image*: hi and lo tiles in the K-major 128-byte-swizzled form that the
// MMA reads from shared memory, 32 K elements by all rows per K block, for
// each of its uses (rows = batch for the activations' products, K = batch for
// the weight gradients).  A product is then bulk copies into a ring, MMAs and
// an epilogue, and nothing else.
//
//   prep     x of the batch -> Xf [rows][n_in], Xt [n_in][rows]
//   act      z = A W^T + b, a = gelu(z): z and the images of a (two launches)
//   mid      out = a2 W3^T + b3, g_out = 2 (out - t) / count (every block of a
//            row tile computes both: 12 MMAs per K block are cheaper than a
//            launch), then g_z2 = (g_out W3) gelu'(z2) for its columns
//   grad     g_z1 = (g_z2 W2) gelu'(z1)
//   dw       dW3, dW2 and dW1 by K ranges, one launch
//   finish   sums of the ranges, column sums for the biases, the loss, Adam,
//            the weights' images and the next batch's prep
//
// Consecutive kernels of a step overlap their prologues (programmatic
// dependent launch): each waits for its predecessor before it touches memory.
// Rows beyond the batch and columns beyond an operand are zeros in the images,
// so no product needs a bounds check.  The weights' images live with the object
// and follow every change of the parameters; those of the batch (nine operands
// of up to kTrainRows rows) are allocated by the first step that wants them, so
// an object that only runs forward does without.  A first step under capture,
// or where they do not fit, takes the generic products (same sums).  Every sum has a fixed order.  Waits are
// bounded; a block whose wait runs out records it and writes nothing.
//
// What bounds it: latency.  A 1,024 x 256 x 256 product is 0.4 GFLOP on 128
// SMs; its launch, first copy, eight K blocks and epilogue follow one another
// (10 us).  So the output tiles are as narrow as fills the SMs (16 columns at
// 1,024 rows and 256 units; 32 cost 2 us more a product, 64 seven), and eight
// epilogue warps share a tile.  A step of 1,024 rows, 221 -> 256 -> 256 -> 4:
// 170 us in 19 launches, 81 in six with four epilogue warps and weights
// updated element by element, 58 so (each kernel's prologue under the end of
// the one before).
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <new>
#include <vector>
#include <cuda_runtime.h>

#include "cg_internal.h"
#include "cg_mlp.h"
#include "cg_tc.cuh"

namespace cg {

// hi (then lo) image of an operand: element (row, k) of K block kb at byte
// kb rows 128 + row 128 + 16 ((k / 4 % 8) ^ (row % 8)) + 4 (k % 4)
struct Img {
    unsigned char* p = nullptr;
    int64_t lo = 0;      // byte offset of the lo image
    int rows = 0;        // rows per K block (a multiple of 128)
};

struct TrainImages {
    int num_sms = 0;
    bool ready = false;          // the batch images are allocated
    bool refused = false;        // they did not fit: the generic products serve
    Img xf, xt, a1f, a1t, a2f, a2t, g3t, g2f, g2t, g1t;   // of the batch
    Img w1f, w2f, w2t, w3f, w3t;                          // of the parameters
    float* ws = nullptr;         // K ranges of dW3, dW2, dW1
    unsigned char *weights = nullptr, *batch = nullptr;   // the images' memory
};

namespace {

constexpr int kTile = kGM * 128;                 // one 128-row tile of a K block
constexpr int kEpiThreads = 256;                 // warps w and w + 4 share 32 rows, taking every other 8 columns
constexpr int kCopyWarp = kEpiThreads / 32;
constexpr int kMmaWarp = kCopyWarp + 1;
constexpr int kTrThreads = 32 * (kMmaWarp + 1);
constexpr int kMaxRing = 6;
constexpr uint32_t kTrPolls = 1u << 22;
constexpr int kFinThreads = 256;

__device__ __forceinline__ uint32_t swz(int row, int k)
{
    return static_cast<uint32_t>(row * 128 + (((((k >> 2) & 7) ^ (row & 7))) << 4) + ((k & 3) << 2));
}

__device__ __forceinline__ void put(const Img& im, int row, int k, float v)
{
    unsigned char* d = im.p + static_cast<int64_t>(k >> 5) * im.rows * 128 + swz(row, k & 31);
    const float h = tf32_rn(v);
    *reinterpret_cast<float*>(d) = h;
    *reinterpret_cast<float*>(d + im.lo) = tf32_rn(v - h);
}
// four consecutive k (k % 4 == 0)
__device__ __forceinline__ void put4(const Img& im, int row, int k, const float* v)
{
    unsigned char* d = im.p + static_cast<int64_t>(k >> 5) * im.rows * 128 + swz(row, k & 31);
    float h[4], l[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        h[i] = tf32_rn(v[i]);
        l[i] = tf32_rn(v[i] - h[i]);
    }
    *reinterpret_cast<float4*>(d) = make_float4(h[0], h[1], h[2], h[3]);
    *reinterpret_cast<float4*>(d + im.lo) = make_float4(l[0], l[1], l[2], l[3]);
}

// bounded wait that also gives up once another thread has set the abort flag
__device__ __forceinline__ bool tr_wait(uint64_t* bar, uint32_t parity, volatile int* abort_flag, bool watch)
{
    const uint64_t t0 = tc::globaltimer_ns();
    for (uint32_t i = 0; i < kTrPolls; ++i) {
        if (tc::mbar_try_wait(bar, parity)) return true;
        if ((i & 255u) == 255u && ((watch && *abort_flag) || tc::globaltimer_ns() - t0 > tc::kWaitLimitNs)) return false;
    }
    return false;
}
__device__ __forceinline__ bool epi_any(bool flag)
{
    uint32_t r;
    asm volatile(
        "{\n .reg .pred p, q;\n setp.ne.u32 p, %1, 0;\n bar.red.or.pred q, 1, %2, p;\n selp.u32 %0, 1, 0, q;\n}\n"
        : "=r"(r)
        : "r"(flag ? 1u : 0u), "n"(kEpiThreads)
        : "memory");
    return r != 0;
}

// A block's shared memory: a ring of operand stages (A hi, A lo, B hi, B lo),
// the barriers and, after them, what a kernel adds.
struct Ring {
    unsigned char* st;
    int stages, bytes;           // stages, bytes of one
    uint64_t *full, *empty, *done;
    uint32_t* tmem_slot;
    volatile int* abort_flag;
};
__host__ __device__ constexpr int ring_stage_bytes(int bn) { return 2 * kTile + 2 * bn * 128; }
constexpr int kRingTail = 256;   // barriers, TMEM slot, flag

__device__ __forceinline__ unsigned char* align1024(unsigned char* p)
{
    return reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(p) + 1023) & ~static_cast<uintptr_t>(1023));
}
__device__ __forceinline__ Ring ring_init(unsigned char* sm, int stages, int bn, int tmem_cols)
{
    Ring r;
    r.st = sm;
    r.stages = stages;
    r.bytes = ring_stage_bytes(bn);
    r.full = reinterpret_cast<uint64_t*>(sm + stages * r.bytes);
    r.empty = r.full + kMaxRing;
    r.done = r.empty + kMaxRing;                       // [3]: done, and two for the kernel
    r.tmem_slot = reinterpret_cast<uint32_t*>(r.done + 3);
    r.abort_flag = reinterpret_cast<volatile int*>(r.tmem_slot + 1);
    if (threadIdx.x == 0) {
        for (int s = 0; s < stages; ++s) {
            tc::mbar_init(&r.full[s], 1);
            tc::mbar_init(&r.empty[s], 1);
        }
        tc::mbar_init(&r.done[0], 1);
        tc::mbar_init(&r.done[1], 1);
        tc::mbar_init(&r.done[2], kGM);
        *r.abort_flag = 0;
        tc::fence_mbar_init();
    }
    if (threadIdx.x >= 32 * kMmaWarp) tc::tmem_alloc(r.tmem_slot, tmem_cols);
    tc::tc_fence_before();
    __syncthreads();
    tc::tc_fence_after();
    return r;
}
__device__ __forceinline__ void ring_end(const Ring& r, int tmem_cols)
{
    tc::tc_fence_before();
    __syncthreads();
    if (threadIdx.x >= 32 * kMmaWarp) {
        __syncwarp();
        tc::tc_fence_after();
        tc::tmem_dealloc(*r.tmem_slot, tmem_cols);
    }
}

// copy warp, one lane: K blocks kb0 .. kb0 + nkb of 128 rows of a and bn rows
// of b into the ring
__device__ __forceinline__ void ring_copy(const Ring& r, const Img& a, int m0, const Img& b, int n0, int bn, int kb0,
                                          int nkb)
{
    int i = 0;
    for (; i < nkb; ++i) {
        const int s = i % r.stages;
        if (i >= r.stages && !tr_wait(&r.empty[s], (i / r.stages - 1) & 1u, r.abort_flag, true)) {
            *r.abort_flag = 1;
            break;
        }
        unsigned char* st = r.st + s * r.bytes;
        const unsigned char* pa = a.p + (static_cast<int64_t>(kb0 + i) * a.rows + m0) * 128;
        const unsigned char* pb = b.p + (static_cast<int64_t>(kb0 + i) * b.rows + n0) * 128;
        const uint32_t nb = static_cast<uint32_t>(bn) * 128u;
        tc::mbar_arrive_expect_tx(&r.full[s], 2u * kTile + 2u * nb);
        tc::bulk_g2s(st, pa, kTile, &r.full[s]);
        tc::bulk_g2s(st + kTile, pa + a.lo, kTile, &r.full[s]);
        tc::bulk_g2s(st + 2 * kTile, pb, nb, &r.full[s]);
        tc::bulk_g2s(st + 2 * kTile + nb, pb + b.lo, nb, &r.full[s]);
    }
    // the last copies of every stage have landed before the block goes on
    for (int q = i > r.stages ? i - r.stages : 0; q < i; ++q)
        (void)tc::mbar_wait(&r.full[q % r.stages], (q / r.stages) & 1u, kTrPolls);
}

// the 12 MMAs of one K block: hi hi, hi lo, lo hi for each eight K elements
__device__ __forceinline__ void mma_block(uint32_t d, uint32_t ah, uint32_t al, uint32_t bh, uint32_t bl,
                                          uint32_t idesc, bool first)
{
#pragma unroll
    for (int kk = 0; kk < kGK / 8; ++kk) {
        const uint32_t ko = kk * 32;
        tc::mma_tf32(d, tc::sdesc_sw128(ah + ko), tc::sdesc_sw128(bh + ko), idesc, (!first || kk > 0) ? 1u : 0u);
        tc::mma_tf32(d, tc::sdesc_sw128(ah + ko), tc::sdesc_sw128(bl + ko), idesc, 1u);
        tc::mma_tf32(d, tc::sdesc_sw128(al + ko), tc::sdesc_sw128(bh + ko), idesc, 1u);
    }
}
// MMA warp, one lane: consume nkb stages into columns d, then commit `done`
__device__ __forceinline__ void ring_mma(const Ring& r, uint32_t d, int bn, int nkb)
{
    const uint32_t idesc = tc::idesc_tf32(kGM, bn);
    for (int i = 0; i < nkb; ++i) {
        const int s = i % r.stages;
        if (!tr_wait(&r.full[s], (i / r.stages) & 1u, r.abort_flag, true)) {
            *r.abort_flag = 1;
            break;
        }
        tc::tc_fence_after();
        const uint32_t ah = tc::smem_u32(r.st + s * r.bytes);
        mma_block(d, ah, ah + kTile, ah + 2 * kTile, ah + 2 * kTile + bn * 128, idesc, i == 0);
        tc::mma_commit(&r.empty[s]);
    }
    tc::mma_commit(&r.done[0]);   // also on abort: TMEM is quiescent before it is read or freed
}
// epilogue threads: wait for `done`; false (the same in every one) on failure
__device__ __forceinline__ bool ring_wait(const Ring& r, uint64_t* done, int* err)
{
    __syncwarp();
    const bool waited = tr_wait(done, 0, r.abort_flag, false);
    const bool failed = epi_any(!waited || *r.abort_flag);
    tc::tc_fence_after();
    if (failed && threadIdx.x == 0 && err) atomicExch(err, 1);
    return !failed;
}

// eight values of a row of the batch, columns c0 .. c0 + 7 (nc of them
// real): images with rows = batch (f) and K = batch (t); zero rows beyond n
__device__ __forceinline__ void put_images(const Img& f, const Img& t, int row, int n, int c0, int nc, float (&v)[8])
{
    if (row >= n)
#pragma unroll
        for (int i = 0; i < 8; ++i) v[i] = 0.f;
    if (f.p) {
        if (nc == 8) {
#pragma unroll
            for (int i = 0; i < 8; i += 4) put4(f, row, c0 + i, v + i);
        } else {
#pragma unroll
            for (int i = 0; i < 8; ++i)
                if (i < nc) put(f, row, c0 + i, v[i]);
        }
    }
#pragma unroll
    for (int i = 0; i < 8; ++i)
        if (i < nc) put(t, c0 + i, row, v[i]);
}
// the same values as a row of an FP32 matrix [n][ld]
__device__ __forceinline__ void put_row(float* m, int ld, int row, int n, int c0, int nc, const float (&v)[8])
{
    if (row >= n) return;
    float* d = m + static_cast<int64_t>(row) * ld + c0;
    if (nc == 8 && (ld & 3) == 0) {
#pragma unroll
        for (int i = 0; i < 8; i += 4) *reinterpret_cast<float4*>(d + i) = make_float4(v[i], v[i + 1], v[i + 2], v[i + 3]);
    } else {
#pragma unroll
        for (int i = 0; i < 8; ++i)
            if (i < nc) d[i] = v[i];
    }
}
__device__ __forceinline__ void get_row(const float* m, int ld, int row, int n, int c0, int nc, float (&v)[8])
{
#pragma unroll
    for (int i = 0; i < 8; ++i) v[i] = 0.f;
    if (row >= n) return;
    const float* d = m + static_cast<int64_t>(row) * ld + c0;
    if (nc == 8 && (ld & 3) == 0) {
#pragma unroll
        for (int i = 0; i < 8; i += 4) {
            const float4 q = *reinterpret_cast<const float4*>(d + i);
            v[i] = q.x;
            v[i + 1] = q.y;
            v[i + 2] = q.z;
            v[i + 3] = q.w;
        }
    } else {
#pragma unroll
        for (int i = 0; i < 8; ++i)
            if (i < nc) v[i] = d[i];
    }
}

// act (GRAD = false): z = a b^T + bias -> fp [n][N], gelu(z) -> the images.
// grad (GRAD = true): g = a b^T gelu'(aux) -> fp [n][N] and the images.
// One block per 128 x bn tile.
struct ProductArgs {
    Img a, b, f, t;
    int n, N, nkb, bn, stages, tmem_cols;
    const float *bias, *aux;
    float* fp;
    int* err;
};
template <bool GRAD>
__global__ void __launch_bounds__(kTrThreads, 1) product_kernel(const __grid_constant__ ProductArgs q)
{
    extern __shared__ __align__(1024) unsigned char tsm_raw[];
    unsigned char* const tsm = align1024(tsm_raw);
    tc::pdl_start();
    const Ring r = ring_init(tsm, q.stages, q.bn, q.tmem_cols);
    tc::pdl_wait();
    const int m0 = blockIdx.y * kGM, n0 = blockIdx.x * q.bn;
    const int ncols = q.N - n0 < q.bn ? q.N - n0 : q.bn, bn = (ncols + 15) & ~15;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t tmem = *r.tmem_slot;
    if (warp == kCopyWarp) {
        if (lane == 0) ring_copy(r, q.a, m0, q.b, n0, bn, 0, q.nkb);
    } else if (warp == kMmaWarp) {
        if (lane == 0) {
            ring_mma(r, tmem, bn, q.nkb);
            (void)tc::mbar_wait(&r.done[0], 0, kTrPolls);
        }
    } else {
        const int row = m0 + 32 * (warp & 3) + lane, c0 = 8 * (warp >> 2);
        float ax[8];
        if (GRAD) get_row(q.aux, q.N, row, q.n, n0 + c0, max(0, min(8, ncols - c0)), ax);   // the first, during the products
        if (ring_wait(r, &r.done[0], q.err)) {
            const uint32_t base = tmem + (static_cast<uint32_t>((warp & 3) * 32) << 16);
            for (int c = c0; c < ncols; c += 16) {
                const int nc = min(8, ncols - c);
                float v[8];
                tc::tmem_ld8(base + c, v);
                if (GRAD) {
                    if (c > c0) get_row(q.aux, q.N, row, q.n, n0 + c, nc, ax);
#pragma unroll
                    for (int i = 0; i < 8; ++i) v[i] *= gelu_grad_f(ax[i]);
                    put_row(q.fp, q.N, row, q.n, n0 + c, nc, v);
                } else {
#pragma unroll
                    for (int i = 0; i < 8; ++i) v[i] += i < nc ? q.bias[n0 + c + i] : 0.f;
                    put_row(q.fp, q.N, row, q.n, n0 + c, nc, v);
#pragma unroll
                    for (int i = 0; i < 8; ++i) v[i] = gelu_f(v[i]);
                }
                put_images(q.f, q.t, row, q.n, n0 + c, nc, v);
            }
        }
    }
    ring_end(r, q.tmem_cols);
}

// mid: out, g_out and this block's columns of g_z2
struct MidArgs {
    Img a2f, w3f, w3t, g3t, g2f, g2t;
    int n, H, no, nkb, bn, stages, tmem_cols;
    const float *b3, *z2, *t;
    const int32_t* perm;
    int64_t n_src;
    float scale;                 // 2 / (n no)
    float *out, *tb, *g_out, *g_z2;
    int* err;
};
__global__ void __launch_bounds__(kTrThreads, 1) mid_kernel(const __grid_constant__ MidArgs q)
{
    extern __shared__ __align__(1024) unsigned char tsm_raw[];
    unsigned char* const tsm = align1024(tsm_raw);
    tc::pdl_start();
    const Ring r = ring_init(tsm, q.stages, 16, q.tmem_cols);
    // after the ring: g_out's tile (A of the second product) and the W3 rows (B)
    unsigned char* ga = tsm + ((q.stages * r.bytes + kRingTail + 1023) & ~1023);   // hi, lo
    unsigned char* wb = ga + 2 * kTile;                                            // hi, lo of bn rows
    tc::pdl_wait();
    const int m0 = blockIdx.y * kGM, n0 = blockIdx.x * q.bn;
    const int ncols = q.H - n0 < q.bn ? q.H - n0 : q.bn, bn = (ncols + 15) & ~15;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t tmem = *r.tmem_slot;
    uint64_t* w_full = &r.empty[kMaxRing - 1];   // (the ring of this kernel is shorter: host)
    if (threadIdx.x == 0) {
        tc::mbar_init(w_full, 1);
        tc::fence_mbar_init();
    }
    __syncthreads();
    if (warp == kCopyWarp) {
        if (lane == 0) {
            const uint32_t nb = static_cast<uint32_t>(bn) * 128u;
            const unsigned char* pw = q.w3t.p + static_cast<int64_t>(n0) * 128;
            tc::mbar_arrive_expect_tx(w_full, 2u * nb);
            tc::bulk_g2s(wb, pw, nb, w_full);
            tc::bulk_g2s(wb + nb, pw + q.w3t.lo, nb, w_full);
            ring_copy(r, q.a2f, m0, q.w3f, 0, 16, 0, q.nkb);
            (void)tc::mbar_wait(w_full, 0, kTrPolls);
        }
    } else if (warp == kMmaWarp) {
        if (lane == 0) {
            ring_mma(r, tmem, 16, q.nkb);
            // the second product: g_out (written by the epilogue threads) times W3
            if (!*r.abort_flag && tr_wait(&r.done[2], 0, r.abort_flag, true) && tr_wait(w_full, 0, r.abort_flag, true)) {
                tc::tc_fence_after();
                const uint32_t a = tc::smem_u32(ga), b = tc::smem_u32(wb);
                mma_block(tmem + 16, a, a + kTile, b, b + bn * 128, tc::idesc_tf32(kGM, bn), true);
            } else {
                *r.abort_flag = 1;
            }
            tc::mma_commit(&r.done[1]);
            (void)tc::mbar_wait(&r.done[1], 0, kTrPolls);
        }
    } else {
        const int rl = 32 * (warp & 3) + lane, row = m0 + rl, c0 = 8 * (warp >> 2);
        const uint32_t base = tmem + (static_cast<uint32_t>((warp & 3) * 32) << 16);
        float ax[8];
        get_row(q.z2, q.H, row, q.n, n0 + c0, max(0, min(8, ncols - c0)), ax);
        float tv[16];
#pragma unroll
        for (int j = 0; j < 16; ++j) tv[j] = 0.f;
        if (warp < 4 && row < q.n) {
            const int64_t src = q.perm ? q.perm[row] : row;
            if (src >= 0 && src < q.n_src)
#pragma unroll
                for (int j = 0; j < 16; ++j)
                    if (j < q.no) tv[j] = q.t[src * q.no + j];
        }
        bool ok = ring_wait(r, &r.done[0], q.err);
        if (warp < 4) {
            float v[16], g[32];
            if (ok) {
                tc::tmem_ld16(base, v);
#pragma unroll
                for (int j = 0; j < 32; ++j) g[j] = 0.f;
#pragma unroll
                for (int j = 0; j < 16; ++j)
                    if (j < q.no) {
                        v[j] += q.b3[j];
                        const float d = v[j] - tv[j];
                        g[j] = row < q.n ? q.scale * d : 0.f;
                    }
                // the tile of g_out as the MMA reads it: this thread's row of 32 K elements
#pragma unroll
                for (int k = 0; k < 32; k += 4) {
                    float h[4], l[4];
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        h[i] = tf32_rn(g[k + i]);
                        l[i] = tf32_rn(g[k + i] - h[i]);
                    }
                    *reinterpret_cast<float4*>(ga + swz(rl, k)) = make_float4(h[0], h[1], h[2], h[3]);
                    *reinterpret_cast<float4*>(ga + kTile + swz(rl, k)) = make_float4(l[0], l[1], l[2], l[3]);
                }
                tc::fence_proxy_async_smem();
                tc::tc_fence_before();
            }
            tc::mbar_arrive(&r.done[2]);
            if (ok && blockIdx.x == 0) {   // one block of the row tile keeps them
#pragma unroll
                for (int j = 0; j < 16; ++j)
                    if (j < q.no) {
                        put(q.g3t, j, row, g[j]);
                        if (row < q.n) {
                            const int64_t o = static_cast<int64_t>(row) * q.no + j;
                            q.out[o] = v[j];
                            q.tb[o] = tv[j];
                            q.g_out[o] = g[j];
                        }
                    }
            }
        }
        if (ok) ok = ring_wait(r, &r.done[1], q.err);
        if (ok)
            for (int c = c0; c < ncols; c += 16) {
                const int nc = min(8, ncols - c);
                float v[8];
                tc::tmem_ld8(base + 16 + c, v);
                if (c > c0) get_row(q.z2, q.H, row, q.n, n0 + c, nc, ax);
#pragma unroll
                for (int i = 0; i < 8; ++i) v[i] *= gelu_grad_f(ax[i]);
                put_row(q.g_z2, q.H, row, q.n, n0 + c, nc, v);
                put_images(q.g2f, q.g2t, row, q.n, n0 + c, nc, v);
            }
    }
    ring_end(r, q.tmem_cols);
}

// dw: one weight-gradient product C[M][N] = a b^T per entry, K range z of the
// tile to ws[z][M][N]
struct DwJob {
    Img a, b;
    int M, N, nkb, kb_per, tiles_n, first;   // first: its first block
    float* ws;
};
struct DwArgs {
    DwJob job[3];
    int bn, stages, tmem_cols;
    int* err;
};
__global__ void __launch_bounds__(kTrThreads, 1) dw_kernel(const __grid_constant__ DwArgs q)
{
    extern __shared__ __align__(1024) unsigned char tsm_raw[];
    unsigned char* const tsm = align1024(tsm_raw);
    tc::pdl_start();
    const Ring r = ring_init(tsm, q.stages, q.bn, q.tmem_cols);
    tc::pdl_wait();
    const int bid = static_cast<int>(blockIdx.x);
    const DwJob& j = bid >= q.job[2].first ? q.job[2] : bid >= q.job[1].first ? q.job[1] : q.job[0];
    const int splits = (j.nkb + j.kb_per - 1) / j.kb_per;
    const int i = bid - j.first, z = i % splits, tile = i / splits;
    const int m0 = (tile / j.tiles_n) * kGM, n0 = (tile % j.tiles_n) * q.bn;
    const int kb0 = z * j.kb_per, nkb = min(j.kb_per, j.nkb - kb0);
    const int ncols = min(q.bn, j.N - n0), bn = (ncols + 15) & ~15;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t tmem = *r.tmem_slot;
    if (warp == kCopyWarp) {
        if (lane == 0) ring_copy(r, j.a, m0, j.b, n0, bn, kb0, nkb);
    } else if (warp == kMmaWarp) {
        if (lane == 0) {
            ring_mma(r, tmem, bn, nkb);
            (void)tc::mbar_wait(&r.done[0], 0, kTrPolls);
        }
    } else if (ring_wait(r, &r.done[0], q.err)) {
        const uint32_t base = tmem + (static_cast<uint32_t>((warp & 3) * 32) << 16);
        const int row = m0 + 32 * (warp & 3) + lane;
        float* ws = j.ws + static_cast<int64_t>(z) * j.M * j.N;
        for (int c = 8 * (warp >> 2); c < ncols; c += 16) {
            float v[8];
            tc::tmem_ld8(base + c, v);
            put_row(ws, j.N, row, j.M, n0 + c, min(8, ncols - c), v);
        }
    }
    ring_end(r, q.tmem_cols);
}

// x rows of a batch into their images, one 32 x 32 tile per call of the block
struct PrepArgs {
    Img xf, xt;
    const float* x;
    const int32_t* perm;
    int64_t n_src;
    int n, ni, tiles_k, tiles;
};
__device__ __forceinline__ void prep_tile(const PrepArgs& q, int tile, float (*buf)[33])
{
    const int r0 = (tile / q.tiles_k) * 32, k0 = (tile % q.tiles_k) * 32;
    const int c = threadIdx.x & 31, y = threadIdx.x >> 5;
#pragma unroll
    for (int i = 0; i < 32; i += kFinThreads / 32) {
        const int row = r0 + y + i, k = k0 + c;
        float v = 0.f;
        if (row < q.n && k < q.ni) {
            const int64_t src = q.perm ? q.perm[row] : row;
            if (src >= 0 && src < q.n_src) v = q.x[src * q.ni + k];
        }
        buf[y + i][c] = v;
        put(q.xf, row, k, v);
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 32; i += kFinThreads / 32) put(q.xt, k0 + y + i, r0 + c, buf[c][y + i]);
    __syncthreads();
}
__global__ void __launch_bounds__(kFinThreads) prep_kernel(const __grid_constant__ PrepArgs q)
{
    __shared__ float buf[32][33];
    tc::pdl_start();
    tc::pdl_wait();
    prep_tile(q, static_cast<int>(blockIdx.x), buf);
}

// finish: block roles by index -- bias columns, loss, weights, next prep
struct FinishArgs {
    float *theta, *grad, *m, *v;
    int64_t np, oW1, ob1, oW2, ob2, oW3, ob3;
    int ni, H, no, n;
    // weight gradients: K ranges to add (null: take grad as it is)
    const float *ws1, *ws2, *ws3;
    int s1, s2, s3;
    const float *g_z1, *g_z2, *g_out, *out, *tb;
    float *loss, *loss_copy;
    int adam;                    // 1: an Adam step
    AdamStep a;
    int images;                  // 1: write the weights' images
    Img w1f, w2f, w2t, w3f, w3t;
    int bias_blocks, loss_block, weight_blocks;
    PrepArgs prep;
};

struct ParamState {
    float th, m, v;
};
__device__ __forceinline__ ParamState load_param(const FinishArgs& q, int64_t i)
{
    return {q.theta[i], q.adam ? q.m[i] : 0.f, q.adam ? q.v[i] : 0.f};
}
__device__ __forceinline__ float finish_param(const FinishArgs& q, int64_t i, float gi, const ParamState& p)
{
    float th = p.th;
    if (q.adam) {
        const float mi = fmaf(q.a.b1, p.m, (1.0f - q.a.b1) * gi);
        const float vi = fmaf(q.a.b2, p.v, (1.0f - q.a.b2) * gi * gi);
        q.m[i] = mi;
        q.v[i] = vi;
        th -= q.a.lr * (mi / q.a.bc1) / (sqrtf(vi / q.a.bc2) + q.a.eps);
        q.theta[i] = th;
    }
    return th;
}

__global__ void __launch_bounds__(kFinThreads) finish_kernel(const __grid_constant__ FinishArgs q)
{
    __shared__ float buf[32][33];
    tc::pdl_start();
    tc::pdl_wait();
    int b = static_cast<int>(blockIdx.x);
    const int t = threadIdx.x;
    if (b < q.bias_blocks) {
        // eight bias gradients: column sums in colsum_kernel's order (rows y,
        // y + 32, ... per partial sum, then the 32 partial sums in order)
        const int cx = t & 7, y = t >> 3;
        const int c = 8 * b + cx, cols = 2 * q.H + q.no;
        const float* g = c < q.H ? q.g_z1 : c < 2 * q.H ? q.g_z2 : q.g_out;
        const int ld = c < 2 * q.H ? q.H : q.no;
        const int col = c < q.H ? c : c < 2 * q.H ? c - q.H : c - 2 * q.H;
        const int64_t i = (c < q.H ? q.ob1 : c < 2 * q.H ? q.ob2 : q.ob3) + col;
        if (q.ws1) {
            float s = 0.f;
            if (c < cols) {
#pragma unroll 16
                for (int r = y; r < q.n; r += 32) s += g[static_cast<int64_t>(r) * ld + col];
            }
            buf[y][cx] = s;
            __syncthreads();
        }
        if (y == 0 && c < cols) {
            float s = 0.f;
            if (q.ws1) {
                s = buf[0][cx];
                for (int k = 1; k < 32; ++k) s += buf[k][cx];
                q.grad[i] = s;
            } else {
                s = q.grad[i];
            }
            finish_param(q, i, s, load_param(q, i));
        }
        return;
    }
    b -= q.bias_blocks;
    if (q.loss_block) {
        if (b == 0) {
            // the loss as mse_kernel and loss_final_kernel sum it: partial p
            // takes elements 256 p + i + 65536 m, a tree over i, then a tree
            // over the partials
            const int64_t count = static_cast<int64_t>(q.n) * q.no;
            const int lane = t & 31;
            float* part = &buf[0][0];
            part[t] = 0.f;
            __syncthreads();
            for (int p = t >> 5; p < kLossBlocks && 256 * p < count; p += kFinThreads / 32) {
                float s[8];
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    const int64_t e = 256 * p + lane + 32 * k;
                    const float d = e < count ? q.out[e] - q.tb[e] : 0.f;
                    s[k] = d * d;
                }
                for (int64_t e0 = 256 * p + lane + 256 * kLossBlocks; e0 < count; e0 += 256 * kLossBlocks)
#pragma unroll
                    for (int k = 0; k < 8; ++k) {
                        const int64_t e = e0 + 32 * k;
                        if (e < count) {
                            const float d = q.out[e] - q.tb[e];
                            s[k] = fmaf(d, d, s[k]);
                        }
                    }
#pragma unroll
                for (int w = 4; w > 0; w >>= 1)
#pragma unroll
                    for (int k = 0; k < w; ++k) s[k] += s[k + w];
#pragma unroll
                for (int w = 16; w > 0; w >>= 1) s[0] += __shfl_down_sync(0xffffffffu, s[0], w);
                if (lane == 0) part[p] = s[0];
            }
            __syncthreads();
            for (int w = 128; w > 0; w >>= 1) {
                if (t < w) part[t] += part[t + w];
                __syncthreads();
            }
            if (t == 0) {
                const float l = part[0] / static_cast<float>(count);
                q.loss[0] = l;
                if (q.loss_copy) q.loss_copy[0] = l;
            }
            return;
        }
        --b;
    }
    if (b < q.weight_blocks) {
        // a 32 x 32 tile of one weight matrix: gradients, Adam and the image
        // by rows, the transposed image through shared memory
        int layer = 1, tiles_k = (q.ni + 31) >> 5, tiles_h = (q.H + 31) >> 5, tile = b;
        if (tile >= tiles_h * tiles_k) {
            tile -= tiles_h * tiles_k;
            layer = 2;
            tiles_k = tiles_h;
            if (tile >= tiles_h * tiles_h) {
                tile -= tiles_h * tiles_h;
                layer = 3;
            }
        }
        const int rows = layer == 3 ? q.no : q.H, cols = layer == 1 ? q.ni : q.H;
        const int r0 = (tile / tiles_k) * 32, k0 = (tile % tiles_k) * 32, c = t & 31, y = t >> 5;
        const int64_t base = layer == 1 ? q.oW1 : layer == 2 ? q.oW2 : q.oW3;
        const float* ws = layer == 1 ? q.ws1 : layer == 2 ? q.ws2 : q.ws3;
        const int splits = !ws ? 0 : layer == 1 ? q.s1 : layer == 2 ? q.s2 : q.s3;
        const int64_t mn = static_cast<int64_t>(rows) * cols;
        // every load goes out before the first is used; the K ranges are
        // added in order
        float part[4][kGMaxSplit];
        ParamState st[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int r = r0 + y + 8 * i, k = k0 + c;
            const bool in = r < rows && k < cols;
            const int64_t e = in ? static_cast<int64_t>(r) * cols + k : 0;
            st[i] = load_param(q, base + e);
#pragma unroll
            for (int z = 0; z < kGMaxSplit; ++z)
                part[i][z] = (ws && z < splits) ? ws[z * mn + e] : (z == 0 ? q.grad[base + e] : 0.f);
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int r = r0 + y + 8 * i, k = k0 + c;
            if (r >= rows || k >= cols) continue;
            float gi = part[i][0];
#pragma unroll
            for (int z = 1; z < kGMaxSplit; ++z)
                if (z < splits) gi += part[i][z];
            const int64_t p = base + static_cast<int64_t>(r) * cols + k;
            if (ws) q.grad[p] = gi;
            const float th = finish_param(q, p, gi, st[i]);
            buf[y + 8 * i][c] = th;
            if (q.images) put(layer == 1 ? q.w1f : layer == 2 ? q.w2f : q.w3f, r, k, th);
        }
        if (q.images && layer > 1) {
            __syncthreads();
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int k = k0 + y + 8 * i, r = r0 + c;
                if (r < rows && k < cols) put(layer == 2 ? q.w2t : q.w3t, k, r, buf[c][y + 8 * i]);
            }
        }
        return;
    }
    b -= q.weight_blocks;
    if (b < q.prep.tiles) prep_tile(q.prep, b, buf);
}

template <class A>
cudaError_t launch_pdl(void (*fn)(A), dim3 grid, int threads, size_t smem, cudaStream_t s, A a)
{
    void* args[] = {&a};
    return launch_dependent(reinterpret_cast<void*>(fn), grid, dim3(threads), args, smem, s);
}

int up(int v, int m) { return (v + m - 1) / m * m; }
int kblocks(int k) { return (k + kGK - 1) / kGK; }

// tile columns: the narrowest of 16, 32, 64, 128 whose tiles fit the SMs once
// (a block's time is its chain of copies and K blocks, so filling the SMs
// matters more than re-reading the A tile)
int tile_cols(int tiles_m, int N, int num_sms)
{
    for (int w = 16; w < 128; w *= 2)
        if (tiles_m * ((N + w - 1) / w) <= num_sms) return w;
    return 128;
}
int tmem_cols(int c)
{
    int w = 32;
    while (w < c) w *= 2;
    return w;
}
int ring_stages(int bn, int nkb, int extra, int most)
{
    const int fit = (227 * 1024 - 1024 - kRingTail - extra) / ring_stage_bytes(bn);
    return std::min({most, nkb, fit});
}

PrepArgs prep_args(const cg_mlp_s* m, const TrainBatch& b)
{
    PrepArgs p{};
    p.xf = m->img->xf;
    p.xt = m->img->xt;
    p.x = b.x;
    p.perm = b.perm;
    p.n_src = b.n_src;
    p.n = b.rows;
    p.ni = m->n_in;
    p.tiles_k = kblocks(m->n_in);
    p.tiles = p.tiles_k * (up(b.rows, kGM) / 32);
    return p;
}

FinishArgs finish_args(cg_mlp_s* m)
{
    const TrainImages& im = *m->img;
    const Offsets o = offsets(m);
    FinishArgs f{};
    f.theta = m->theta;
    f.grad = m->grad;
    f.m = m->m;
    f.v = m->v;
    f.np = m->np;
    f.oW1 = o.W1;
    f.ob1 = o.b1;
    f.oW2 = o.W2;
    f.ob2 = o.b2;
    f.oW3 = o.W3;
    f.ob3 = o.b3;
    f.ni = m->n_in;
    f.H = m->H;
    f.no = m->n_out;
    f.images = 1;
    f.w1f = im.w1f;
    f.w2f = im.w2f;
    f.w2t = im.w2t;
    f.w3f = im.w3f;
    f.w3t = im.w3t;
    const int th = (m->H + 31) / 32;
    f.weight_blocks = th * ((m->n_in + 31) / 32 + th + 1);   // 32 x 32 tiles of W1, W2 and W3
    return f;
}

}  // namespace

namespace {

struct ImgShape {
    Img* im;
    int rows, k;
};
// zeroed memory for some images (padding stays zero)
template <int N>
cudaError_t alloc_images(const ImgShape (&all)[N], unsigned char** pool, cudaStream_t s)
{
    int64_t bytes = 0;
    for (const ImgShape& a : all) {
        a.im->rows = up(a.rows, kGM);
        a.im->lo = static_cast<int64_t>(kblocks(a.k)) * a.im->rows * 128;
        bytes += 2 * a.im->lo;
    }
    cudaError_t e = cudaMalloc(pool, bytes);
    if (e == cudaSuccess) e = cudaMemsetAsync(*pool, 0, bytes, s);
    if (e != cudaSuccess) return e;
    unsigned char* p = *pool;
    for (const ImgShape& a : all) {
        a.im->p = p;
        p += 2 * a.im->lo;
    }
    return cudaSuccess;
}

void free_batch_images(TrainImages* im)
{
    if (im->batch) cudaFree(im->batch);
    if (im->ws) cudaFree(im->ws);
    im->batch = nullptr;
    im->ws = nullptr;
}

}  // namespace

cudaError_t train_create(cg_mlp_s* m)
{
    TrainImages* im = new (std::nothrow) TrainImages;
    if (!im) return cudaErrorMemoryAllocation;
    m->img = im;
    cudaError_t e = cudaDeviceGetAttribute(&im->num_sms, cudaDevAttrMultiProcessorCount, m->device);
    if (e != cudaSuccess) return e;
    const int ni = m->n_in, H = m->H, no = m->n_out;
    const ImgShape all[] = {{&im->w1f, H, ni}, {&im->w2f, H, H}, {&im->w2t, H, H}, {&im->w3f, no, H}, {&im->w3t, H, no}};
    if ((e = alloc_images(all, &im->weights, nullptr)) != cudaSuccess) return e;
    const int most = 227 * 1024;
    for (void* fn : {reinterpret_cast<void*>(&product_kernel<false>), reinterpret_cast<void*>(&product_kernel<true>),
                     reinterpret_cast<void*>(&mid_kernel), reinterpret_cast<void*>(&dw_kernel)})
        if ((e = raise_smem_limit(fn, most)) != cudaSuccess) return e;
    return train_refresh(m, nullptr);
}

cudaError_t train_ready(cg_mlp_s* m, int rows, cudaStream_t s, bool* ready)
{
    TrainImages* im = m->img;
    *ready = im->ready && rows <= kTrainRows;
    if (im->ready || im->refused || rows > kTrainRows) return cudaSuccess;
    cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
    cudaError_t e = cudaStreamIsCapturing(s, &st);
    if (e != cudaSuccess || st != cudaStreamCaptureStatusNone) return e;
    // (allocation does not disturb another thread's capture in relaxed mode)
    cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
    if ((e = cudaThreadExchangeStreamCaptureMode(&mode)) != cudaSuccess) return e;
    const int ni = m->n_in, H = m->H, no = m->n_out, B = up(std::min(m->max_batch, kTrainRows), kGM);
    const ImgShape all[] = {{&im->xf, B, ni}, {&im->xt, ni, B}, {&im->a1f, B, H}, {&im->a1t, H, B}, {&im->a2f, B, H},
                            {&im->a2t, H, B}, {&im->g3t, no, B}, {&im->g2f, B, H}, {&im->g2t, H, B}, {&im->g1t, H, B}};
    e = cudaMalloc(&im->ws, sizeof(float) * kGMaxSplit * H * (static_cast<int64_t>(ni) + H + no));
    if (e == cudaSuccess) e = alloc_images(all, &im->batch, s);
    if (e == cudaErrorMemoryAllocation) {
        (void)cudaGetLastError();
        free_batch_images(im);
        im->refused = true;
        e = cudaSuccess;
    } else if (e == cudaSuccess) {
        *ready = im->ready = true;
    }
    (void)cudaThreadExchangeStreamCaptureMode(&mode);
    return e;
}

void train_destroy(cg_mlp_s* m)
{
    if (!m->img) return;
    free_batch_images(m->img);
    if (m->img->weights) cudaFree(m->img->weights);
    delete m->img;
    m->img = nullptr;
}

cudaError_t train_refresh(cg_mlp_s* m, cudaStream_t s)
{
    FinishArgs f = finish_args(m);
    return launch_pdl(finish_kernel, dim3(f.weight_blocks), kFinThreads, 0, s, f);
}

cudaError_t train_adam(cg_mlp_s* m, const AdamStep& a, cudaStream_t s)
{
    FinishArgs f = finish_args(m);
    f.bias_blocks = (2 * m->H + m->n_out + 7) / 8;
    f.adam = 1;
    f.a = a;
    return launch_pdl(finish_kernel, dim3(f.bias_blocks + f.weight_blocks), kFinThreads, 0, s, f);
}

cudaError_t train_prepare(cg_mlp_s* m, const TrainBatch& b, cudaStream_t s)
{
    const PrepArgs p = prep_args(m, b);
    return launch_pdl(prep_kernel, dim3(p.tiles), kFinThreads, 0, s, p);
}

cudaError_t train_step(cg_mlp_s* m, const TrainBatch& b, float* loss_copy, const AdamStep* adam,
                       const TrainBatch* next, cudaStream_t s)
{
    const TrainImages& im = *m->img;
    const Offsets o = offsets(m);
    const int n = b.rows, H = m->H, ni = m->n_in, no = m->n_out;
    const int tiles_m = (n + kGM - 1) / kGM;
    const int w = tile_cols(tiles_m, H, im.num_sms);
    const dim3 grid((H + w - 1) / w, tiles_m);
    cudaError_t e = cudaSuccess;
    auto product = [&](bool grad, const Img& a, const Img& bi, int K, const Img& f, const Img& t, const float* bias,
                       const float* aux, float* fp) {
        ProductArgs q{a, bi, f, t, n, H, kblocks(K), w, 0, tmem_cols(w), bias, aux, fp, m->err};
        q.stages = ring_stages(w, q.nkb, 0, kMaxRing);
        const size_t smem = static_cast<size_t>(q.stages) * ring_stage_bytes(w) + kRingTail + 1024;
        return grad ? launch_pdl(product_kernel<true>, grid, kTrThreads, smem, s, q)
                    : launch_pdl(product_kernel<false>, grid, kTrThreads, smem, s, q);
    };
    e = product(false, im.xf, im.w1f, ni, im.a1f, im.a1t, m->theta + o.b1, nullptr, m->z1);
    if (e == cudaSuccess) e = product(false, im.a1f, im.w2f, H, im.a2f, im.a2t, m->theta + o.b2, nullptr, m->z2);
    if (e != cudaSuccess) return e;
    {
        MidArgs q{im.a2f, im.w3f, im.w3t, im.g3t, im.g2f, im.g2t};
        q.n = n;
        q.H = H;
        q.no = no;
        q.nkb = kblocks(H);
        q.bn = w;
        q.tmem_cols = tmem_cols(16 + w);
        q.b3 = m->theta + o.b3;
        q.z2 = m->z2;
        q.t = b.t;
        q.perm = b.perm;
        q.n_src = b.n_src;
        q.scale = 2.0f / static_cast<float>(static_cast<int64_t>(n) * no);
        q.out = m->out;
        q.tb = m->tb;
        q.g_out = m->g_out;
        q.g_z2 = m->g_z2;
        q.err = m->err;
        const int extra = 1024 + 2 * kTile + 2 * w * 128;
        q.stages = ring_stages(16, q.nkb, extra, kMaxRing - 1);
        const size_t smem = ((q.stages * ring_stage_bytes(16) + kRingTail + 1023) & ~1023) + extra;
        if ((e = launch_pdl(mid_kernel, grid, kTrThreads, smem, s, q)) != cudaSuccess) return e;
    }
    e = product(true, im.g2f, im.w2t, H, Img{}, im.g1t, nullptr, m->z1, m->g_z1);
    if (e != cudaSuccess) return e;
    // weight gradients, K ranges as the generic product splits them
    const SplitRule r3 = split_rule(no, H, n, true), r2 = split_rule(H, H, n, true), r1 = split_rule(H, ni, n, true);
    float* ws3 = im.ws;
    float* ws2 = ws3 + static_cast<int64_t>(kGMaxSplit) * no * H;
    float* ws1 = ws2 + static_cast<int64_t>(kGMaxSplit) * H * H;
    {
        const int nkb = kblocks(n);
        DwArgs q{{{im.g3t, im.a2t, no, H, nkb, r3.kb_per, 0, 0, ws3},
                  {im.g2t, im.a1t, H, H, nkb, r2.kb_per, 0, 0, ws2},
                  {im.g1t, im.xt, H, ni, nkb, r1.kb_per, 0, 0, ws1}}};
        int blocks = 0, longest = 1;
        for (q.bn = 16; q.bn <= 128; q.bn += 16) {   // the narrowest tile whose blocks fit the SMs once
            blocks = 0;
            for (DwJob& j : q.job) {
                j.tiles_n = (j.N + q.bn - 1) / q.bn;
                j.first = blocks;
                blocks += ((j.M + kGM - 1) / kGM) * j.tiles_n * ((nkb + j.kb_per - 1) / j.kb_per);
                longest = std::max(longest, j.kb_per);
            }
            if (blocks <= im.num_sms || q.bn == 128) break;
        }
        q.stages = ring_stages(q.bn, longest, 0, kMaxRing);
        q.tmem_cols = tmem_cols(q.bn);
        q.err = m->err;
        const size_t smem = static_cast<size_t>(q.stages) * ring_stage_bytes(q.bn) + kRingTail + 1024;
        if ((e = launch_pdl(dw_kernel, dim3(blocks), kTrThreads, smem, s, q)) != cudaSuccess) return e;
    }
    FinishArgs f = finish_args(m);
    f.n = n;
    f.ws1 = ws1;
    f.ws2 = ws2;
    f.ws3 = ws3;
    f.s1 = r1.splits;
    f.s2 = r2.splits;
    f.s3 = r3.splits;
    f.g_z1 = m->g_z1;
    f.g_z2 = m->g_z2;
    f.g_out = m->g_out;
    f.out = m->out;
    f.tb = m->tb;
    f.loss = m->loss;
    f.loss_copy = loss_copy;
    f.bias_blocks = (2 * H + no + 7) / 8;
    f.loss_block = 1;
    f.images = adam ? 1 : 0;
    if (adam) {
        f.adam = 1;
        f.a = *adam;
    }
    if (next) f.prep = prep_args(m, *next);
    return launch_pdl(finish_kernel, dim3(f.bias_blocks + 1 + f.weight_blocks + f.prep.tiles), kFinThreads, 0, s, f);
}

}  // namespace cg
