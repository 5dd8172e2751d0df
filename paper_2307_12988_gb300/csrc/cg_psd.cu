// cg_psd.cu -- displacement power spectral density of the fitted-centre
// series and the fit of the mechanical resonance (f0, Q) to it (paper,
// "Experimental Results", Fig. 6: PSDs for 1 s, 10 s and 10 min of data and
// the resonance frequency and quality factor fitted to them).
//
// PSD: Welch's method -- segments of M = 2L samples advanced by L, segment
// mean removed, periodic Hann window, |rfft|^2 averaged over the complete
// segments, one-sided density (factor 2 except at DC and M/2) / (fs sum w^2).
// psd_welch_kernel<L>: one segment per group of L/32 threads; the segment's L
// packed complex values z_n = x_2n + i x_2n+1 are transformed in place in
// shared memory (radix 16, and one smaller radix); the real-FFT split
// X_k = E_k + W_M^k O_k gives |X_k|^2 for k = 0..L, which the threads add up
// in FP64, row by row in the order of the segments; psd_reduce_kernel adds the
// rows in order and scales them.
//
// Resonance: S(f) = A f0^4 / ((f0^2 - f^2)^2 + (f f0 / Q)^2) + B fitted to
// ln S over the bins of a band by Levenberg-Marquardt in FP64 (one cluster of
// eight blocks shares the per-point work, each takes the 4x4 solve);
// initial values from the band (largest bin, smallest bin, half-height
// width); standard errors from diag(H^-1) chi^2 / (n - 4).
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <vector>
#include <cuda_runtime.h>

#include "cg_fft.cuh"
#include "cg_internal.h"
#include "cg_stage.cuh"
#include "cg_tc.cuh"

namespace cg {
constexpr int kWelchThreads = 512;   // threads of a block of the Welch kernel
}

struct cg_psd_s {
    int device = 0;
    int L = 0;                 // complex transform length (M / 2)
    int blocks = 0;            // blocks of the Welch kernel at most
    int rows = 0;              // rows of sums of a block
    size_t smem = 0;
    double sum_w2 = 0.0;       // sum of the squared window
    float* win = nullptr;      // [M / 2 + 1] the window's first half (it is symmetric)
    float2* tw = nullptr;      // the kernel's twiddles (WelchTables)
    int2* pair0 = nullptr;     // [L / 32] buffer places of the last pair of each thread
    int* bin = nullptr;        // [L + 1] PSD bin of each slot of a row of part
    double* part = nullptr;    // [blocks * rows][L + 1] sums of |X_k|^2
};

namespace cg {

namespace {

// The transform of one segment: L = 16 * 16 * R3 * R4 complex points, by a
// group of L / 32 threads (each 32 points).
template <int L>
struct Welch {
    static constexpr int NT = L / 32;                   // threads of a group
    static constexpr int G = kWelchThreads / NT;        // groups of a block
    // The segments s = r, r + R, r + 2 R, ... of row r (R rows) are added up one
    // after another; S groups of a block transform S of them at a time, and
    // each keeps the sums of a 1 / S of the row's bins.
    static constexpr int ROWS = L == 2048 ? 2 : 1;      // rows of a block
    static constexpr int S = G / ROWS;                  // groups of a row: 4, 4, 2, 1
    static constexpr int SL = 32 / S;                   // bins whose sums a thread keeps
    static constexpr int R3 = L == 2048 ? 8 : 16;
    static constexpr int R4 = L / (256 * R3);           // 1, 1, 2, 4
    static constexpr int B = L / 16;                    // points of one first-digit block
    static constexpr int M = 2 * L;
    // twiddle tables, float2 entries, in the order the threads read them
    static constexpr int kT2 = 0;                       // [15][16]      W_256^(r k1)
    static constexpr int kT3 = kT2 + 15 * 16;           // [R3 - 1][256] W_(256 R3)^(r (k1 + 16 k2)), k1 slowest
    static constexpr int kT4 = kT3 + (R3 - 1) * 256;    // [R4 - 1][L / R4] W_L^(r k), by position
    static constexpr int kSplit = kT4 + (R4 - 1) * (L / R4);   // [16][NT] W_M^k of a thread's 16 bin pairs
    static constexpr int kHalf = kSplit + L / 2;        // W_M^(L / 2)
    static constexpr int kTables = kHalf + 1;
    // shared memory: the groups' points, the tables of stages 2 and 3, half
    // the window, |X_k|^2 of the bins that other groups of the row add up,
    // warp sums, mean and middle bin of each group, two barriers of each
    static constexpr int kSmemZ = G * L * 8;
    static constexpr int kSmemT = kSmemZ + (15 * 16 + (R3 - 1) * 256) * 8;
    static constexpr int kSmemX = kSmemT + (M / 2 + 4) * 4;
    static constexpr int kSmemW = kSmemX + G * (S - 1) * SL * NT * 4;
    static constexpr int kSmemB = kSmemW + G * (2 * NT / 32) * 4 + G * 8;
    static constexpr int kSmem = kSmemB + G * 16;
};

struct PsdArgs {
    const float* x;
    int64_t stride;            // elements between consecutive samples
    int64_t K;                 // segments
    int rows;                  // rows of sums
    int vec2;                  // sample pairs are 8-byte aligned and contiguous
    int bulk;                  // so are whole segments, 16-byte aligned
    const float* win;
    const float2* tw;
    const int2* pair0;
    double* part;
};

// Shared-memory place of point p: its low four bits XORed with the next four.
// Every stage's accesses of a half warp then fall on distinct banks (the
// strides of the stages are 2 NT, L / 256, R4 and 1).  The map is linear over
// XOR, so a butterfly computes the address of its first point and reaches the
// others (p ^ d with d disjoint from p, known at compile time) by an XOR with
// a constant and the instruction's immediate offset.
__host__ __device__ constexpr int zsw(int p) { return p ^ ((p >> 4) & 15); }
__device__ __forceinline__ uint32_t zat(uint32_t a, int d)
{
    return (a ^ static_cast<uint32_t>((zsw(d) & 15) << 3)) + static_cast<uint32_t>((d & ~15) << 3);
}
__device__ __forceinline__ float2 zld(uint32_t a)
{
    float2 v;
    asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];\n" : "=f"(v.x), "=f"(v.y) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ void zst(uint32_t a, float2 v)
{
    asm volatile("st.shared.v2.f32 [%0], {%1, %2};\n" ::"r"(a), "f"(v.x), "f"(v.y) : "memory");
}

template <int NT>
__device__ __forceinline__ void group_sync(int g)
{
    asm volatile("bar.sync %0, %1;\n" ::"r"(g + 1), "n"(NT) : "memory");
}

// the S groups of a row
template <int NT, int S>
__device__ __forceinline__ void row_sync(int row, int g)
{
    if constexpr (S == 1)
        group_sync<NT>(g);
    else
        asm volatile("bar.sync %0, %1;\n" ::"r"(9 + row), "n"(S * NT) : "memory");
}

// p = |X|^2 as a double.  A normal p by integer operations: the conversion
// runs on the FP64 pipe, which additions alone keep busy at 1.7 lanes a cycle
// and SM (with conversions 1.2; converted under a predicate 0.9).
__device__ __forceinline__ bool is_normal(float p) { return __float_as_uint(p) - 0x00800000u < 0x7f000000u; }
__device__ __forceinline__ double widen(float p)
{
    const uint32_t u = __float_as_uint(p);
    return __hiloint2double(static_cast<int>((u >> 3) + 0x38000000u), static_cast<int>(u << 29));
}

// Welch sums.  One segment per group of NT threads, its L packed complex
// values z_n = x_2n + i x_2n+1 in shared memory.  The transform runs in place
// (digit-reversed result): the points of a butterfly go back where they were
// read, so a thread needs no barrier between its reads and its writes, and
// after the first stage (stride L / 16) all remaining butterflies of a warp
// stay inside the warp's own 1,024 points: 16 live values per thread.  That
// leaves the registers for the sums of |X_k|^2: the thread that holds bins k
// and L - k (one split, two bins from the same two points and twiddle) adds
// them up over all its segments.
//
// The sums are FP64 and have one order: segment after segment within a row,
// then row after row.  (The fit of a resonance takes or leaves its last step by
// the last bit of chi^2, so a density that differs by 1e-15 can move the fitted
// values by 1e-8.)  Where several groups share a row, each hands |X_k|^2 of the
// bins that another adds up to it through shared memory.
//
// What bounds it: the FP64 additions (16,384 a 32,768-sample segment at 1.7
// lanes a cycle and SM: 9,700 of its 30,000 cycles) and shared-memory traffic
// (1.3 MB, 10,000 cycles).  The samples come by bulk copies in two parts, the
// first under the second half of the split, the second under the additions; the
// last stage's twiddles are requested at once and the split's before its
// barrier (they come from L2).  600 million samples in segments of 32,768: 3.53
// ms, of 16,384 3.74, of 8,192 3.13, of 4,096 3.10 (7.6, 6.3, 5.8 and 4.3 with
// two barriers a stage, sums in L2 and conversions on the FP64 pipe).
template <int L>
__global__ void __launch_bounds__(kWelchThreads, 1) psd_welch_kernel(PsdArgs a)
{
    using W = Welch<L>;
    constexpr int NT = W::NT, R3 = W::R3, R4 = W::R4, B = W::B, M = W::M, G = W::G, S = W::S, SL = W::SL;
    tc::pdl_start();
    extern __shared__ __align__(1024) unsigned char psm[];
    const int g = threadIdx.x / NT, t = threadIdx.x % NT, w = t >> 5, lane = t & 31;
    const uint32_t z = static_cast<uint32_t>(__cvta_generic_to_shared(psm)) + g * L * 8;
    float2* const ts = reinterpret_cast<float2*>(psm + W::kSmemZ);
    const float2* const t2 = ts + W::kT2;
    const float2* const t3 = ts + W::kT3;
    float* const win = reinterpret_cast<float*>(psm + W::kSmemT);
    float* const xch = reinterpret_cast<float*>(psm + W::kSmemX);   // [G][S - 1][SL][NT]
    float* const red = reinterpret_cast<float*>(psm + W::kSmemW) + g * (2 * NT / 32);
    float* const means = reinterpret_cast<float*>(psm + W::kSmemW + G * (2 * NT / 32) * 4);   // [G]
    float* const halfs = means + G;                                                          // [G] |X_(L / 2)|^2
    // group q of the S that share row `row`: its segments are first, first + S R, ...
    const int rr = g / S, q = g % S;
    const int64_t R = a.rows;
    const int64_t row = static_cast<int64_t>(rr) * gridDim.x + blockIdx.x;
    const int64_t nslot = S * R;
    const int64_t first = (row < R ? row : a.K) + q * R;
    // rounds of the row: while its group 0 has a segment
    const uint32_t zt = z + 8 * zsw(t);             // point t, and NT - 1 - t
    const uint32_t zr = z + 8 * zsw(NT - 1 - t);
    const uint32_t zl = z + 8 * t;                  // point t of the samples

    // The samples of a segment lie in the order of its points (the stages'
    // places are those of their 16-point block, permuted).  Contiguous ones
    // come by bulk copies in two parts, as the split of the segment before
    // leaves the blocks they go to: 0 to 4 and 12 to 15, then 5 to 11.
    uint64_t* const bars = reinterpret_cast<uint64_t*>(psm + W::kSmemB) + 2 * g;
    auto stage_part = [&](int64_t s, int part) {   // (one thread)
        const float* x = a.x + s * static_cast<int64_t>(L);
        tc::fence_proxy_async_smem();   // the places were read before they are written
        tc::mbar_arrive_expect_tx(&bars[part], (part ? 7 : 9) * B * 8);
        auto blocks = [&](int b0, int n) {
            tc::bulk_g2s(psm + g * L * 8 + b0 * B * 8, x + 2 * b0 * B, n * B * 8, &bars[part]);
        };
        if (part) {
            blocks(5, 7);
        } else {
            blocks(0, 5);
            blocks(12, 4);
        }
    };
    auto stage_x = [&](int64_t s) {   // the thread's own 32 points of segment s, asynchronously
        const float* x = a.x + s * static_cast<int64_t>(L) * a.stride;
        if (a.vec2) {
            x += 2 * t;
#pragma unroll 8
            for (int i = 0; i < 32; ++i)
                asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(zl + 8 * NT * i), "l"(x + 2 * NT * i) : "memory");
        } else {
            x += 2 * t * a.stride;
#pragma unroll 4
            for (int i = 0; i < 32; ++i) {
                const float* p = x + 2 * NT * i * a.stride;
                asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(zl + 8 * NT * i), "l"(p) : "memory");
                asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(zl + 8 * NT * i + 4), "l"(p + a.stride) : "memory");
            }
        }
        cp_async_commit();
    };
    if (t == 0) {
        tc::mbar_init(&bars[0], 1);
        tc::mbar_init(&bars[1], 1);
        tc::fence_mbar_init();
    }
    if (first < a.K) {
        if (!a.bulk) {
            stage_x(first);
        } else if (t == 0) {
            stage_part(first, 0);
            stage_part(first, 1);
        }
    }
    for (int i = threadIdx.x; i < W::kT4; i += kWelchThreads) ts[i] = a.tw[i];
    for (int i = threadIdx.x; i <= M / 2; i += kWelchThreads) win[i] = a.win[i];
    const int2 p15 = a.pair0[t];
    double acc[SL];   // sums of slots q SL ..; slot 2 i + h is bin h of the thread's pair i
#pragma unroll
    for (int j = 0; j < SL; ++j) acc[j] = 0.0;
    double half = 0.0;   // bin L / 2 (thread 0 of group 0 of the row)
    __syncthreads();

    uint32_t phase = 0;
    bool landed = true;   // (a copy that never does leaves the sums undefined)
    for (int64_t s = first; s - q * R < a.K; s += nslot, phase ^= 1u) {
        const bool live = S == 1 || s < a.K;   // (a row's last round may not need all of its groups)
        float2 tws[16];   // the split's twiddles
        if (live) {
            // the next segment into L2 meanwhile
            if (a.bulk) {
                if (s + nslot < a.K && t == 0) tc::prefetch_l2_bulk(a.x + (s + nslot) * static_cast<int64_t>(L), M * 4);
            } else if (s + nslot < a.K && a.stride <= 4) {
                const char* nx = reinterpret_cast<const char*>(a.x + (s + nslot) * static_cast<int64_t>(L) * a.stride);
                for (int64_t i = t; i < M * a.stride / 32; i += NT) asm volatile("prefetch.global.L2 [%0];\n" ::"l"(nx + 128 * i));
            }
            if (a.bulk)
                landed = landed && tc::mbar_wait(&bars[0], phase, 1u << 24);
            else
                cp_async_wait_all();   // own points only: no barrier
            // ---- segment mean: FP32 sums of 32 samples per first-stage column ----
            float sum[2] = {0.f, 0.f};
            auto column = [&](int r) {
#pragma unroll
                for (int b = 0; b < 2; ++b) {
                    const float2 v = zld(zl + 8 * NT * (b + 2 * r));
                    sum[b] += v.x + v.y;
                }
            };
#pragma unroll
            for (int r = 0; r < 5; ++r) column(r);
            if (a.bulk) landed = landed && tc::mbar_wait(&bars[1], phase, 1u << 24);
#pragma unroll
            for (int r = 5; r < 16; ++r) column(r);
#pragma unroll
            for (int b = 0; b < 2; ++b) {
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) sum[b] += __shfl_xor_sync(0xffffffffu, sum[b], o);
                if (lane == 0) red[w + (NT / 32) * b] = sum[b];
            }
            group_sync<NT>(g);
            if (w == 0) {   // one warp adds the warp sums in FP64
                double tot = lane < 2 * NT / 32 ? static_cast<double>(red[lane]) : 0.0;
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) tot += __shfl_xor_sync(0xffffffffu, tot, o);
                if (lane == 0) means[g] = static_cast<float>(tot / M);
            }
            group_sync<NT>(g);
            const float mean = landed ? means[g] : __int_as_float(0x7fffffff);
            // ---- stage 1: subtract the mean, window, 16 points at stride B ----
#pragma unroll 1
            for (int b = 0; b < 2; ++b) {
                const int j = t + NT * b;
                const uint32_t zj = zat(zt, NT) * b + zt * (1 - b);
                float2 v[16];
#pragma unroll
                for (int r = 0; r < 16; ++r) {
                    const int n = j + r * B;
                    v[r] = zld(zl + 8 * (NT * b + r * B));
                    float2 wn;
                    if (r < 8)
                        wn = *reinterpret_cast<const float2*>(win + 2 * n);
                    else
                        wn = make_float2(win[M - 2 * n], win[M - 2 * n - 1]);
                    v[r] = make_float2((v[r].x - mean) * wn.x, (v[r].y - mean) * wn.y);
                }
                __syncwarp();   // (the points' places lie among those the warp has read)
                Dft<16>::run(v);
#pragma unroll
                for (int r = 0; r < 16; ++r) zst(zat(zj, r * B), v[r]);
            }
            group_sync<NT>(g);
            // ---- stage 2: stride B / 16, inside the warp's 1,024 points from here on ----
#pragma unroll 1
            for (int b = 0; b < 2; ++b) {
                const int be = lane + 32 * b;
                const int base = 1024 * w + (be / (B / 16)) * B + be % (B / 16);
                const int k1 = base / B;
                const uint32_t zb = z + 8 * zsw(base);
                float2 v[16];
#pragma unroll
                for (int r = 0; r < 16; ++r) v[r] = zld(zat(zb, r * (B / 16)));
#pragma unroll
                for (int r = 1; r < 16; ++r) v[r] = cmul(v[r], t2[(r - 1) * 16 + k1]);
                Dft<16>::run(v);
#pragma unroll
                for (int r = 0; r < 16; ++r) zst(zat(zb, r * (B / 16)), v[r]);
            }
            __syncwarp();
            // ---- stage 3: stride R4 ----
#pragma unroll 1
            for (int b = 0; b < 32 / R3; ++b) {
                const int be = lane + 32 * b;
                const int base = 1024 * w + (be / R4) * (R3 * R4) + be % R4;
                const int cg = base / (R3 * R4);
                const uint32_t zb = z + 8 * zsw(base);
                float2 v[R3];
#pragma unroll
                for (int r = 0; r < R3; ++r) v[r] = zld(zat(zb, r * R4));
#pragma unroll
                for (int r = 1; r < R3; ++r) v[r] = cmul(v[r], t3[(r - 1) * 256 + cg]);
                Dft<R3>::run(v);
#pragma unroll
                for (int r = 0; r < R3; ++r) zst(zat(zb, r * R4), v[r]);
            }
            // ---- stage 4: stride 1 ----
            if constexpr (R4 > 1) {
                __syncwarp();
                const float2* t4 = a.tw + W::kT4 + (1024 / R4) * w + lane;
#pragma unroll
                for (int b = 0; b < 32 / R4; ++b) {
                    const uint32_t zb = z + 8 * zsw(1024 * w + R4 * (lane + 32 * b));
                    float2 v[R4];
#pragma unroll
                    for (int r = 0; r < R4; ++r) v[r] = zld(zat(zb, r));
#pragma unroll
                    for (int r = 1; r < R4; ++r) v[r] = cmul(v[r], __ldg(&t4[(r - 1) * (L / R4) + 32 * b]));
                    Dft<R4>::run(v);
#pragma unroll
                    for (int r = 0; r < R4; ++r) zst(zat(zb, r), v[r]);
                }
            }
            // requested ahead of the barrier
            tws[15] = __ldg(&a.tw[W::kSplit + 15 * NT + t]);
#pragma unroll
            for (int i = 0; i < 8; ++i) tws[i] = __ldg(&a.tw[W::kSplit + i * NT + t]);
        }
        row_sync<NT, S>(rr, g);   // (and the other groups have read xch)
        // ---- real-FFT split of bins k and L - k, |X|^2 into the sums ----
        const bool more = s + nslot < a.K;
        float own[SL];   // |X|^2 of the slots that this group adds up
        auto split = [&](int i) {
            const int k1 = i < 14 ? 1 + (i >> 1) : 8, h = i < 14 ? i & 1 : 0;
            const float2 Zb = zld(i < 15 ? zat(zt, k1 * B + NT * h) : z + 8 * p15.x);
            const float2 Zr = zld(i < 15 ? zat(zr, (16 - k1) * B + NT * (1 - h)) : z + 8 * p15.y);
            const float2 E = make_float2(0.5f * (Zb.x + Zr.x), 0.5f * (Zb.y - Zr.y));
            const float2 Dd = make_float2(0.5f * (Zb.x - Zr.x), 0.5f * (Zb.y + Zr.y));
            const float2 C = cmul(tws[i], make_float2(Dd.y, -Dd.x));
            // X_k = E + C; X_(L - k) = conj(E - C), since W_M^(L - k) = -conj W_M^k
            const float2 X = cadd(E, C), Y = csub(E, C);
            const float v[2] = {fmaf(X.x, X.x, X.y * X.y), fmaf(Y.x, Y.x, Y.y * Y.y)};
#pragma unroll
            for (int b = 0; b < 2; ++b) {
                const int slot = 2 * i + b, owner = slot / SL;
                if (S == 1 || owner == q)
                    own[slot % SL] = v[b];
                else
                    xch[((g * (S - 1) + (owner < q ? owner : owner - 1)) * SL + slot % SL) * NT + t] = v[b];
            }
        };
        if (live) {
            // blocks 0 to 4 and 12 to 15 first: the next segment's samples follow
            split(15);
#pragma unroll
            for (int i = 0; i < 8; ++i) split(i);
#pragma unroll
            for (int i = 8; i < 15; ++i) tws[i] = __ldg(&a.tw[W::kSplit + i * NT + t]);
            if (t == 0) {   // bin L / 2 pairs with itself
                constexpr int kPos = R4 > 1 ? R4 / 2 : R3 / 2;   // its last digit is R / 2, the others 0
                const float2 Zh = zld(z + 8 * zsw(kPos));
                const float2 X = cadd(make_float2(Zh.x, 0.f), cmul(__ldg(&a.tw[W::kHalf]), make_float2(Zh.y, -0.f)));
                halfs[g] = fmaf(X.x, X.x, X.y * X.y);
            }
            if (a.bulk) {
                group_sync<NT>(g);
                if (more && t == 0) stage_part(s + nslot, 0);
            }
#pragma unroll
            for (int i = 8; i < 15; ++i) split(i);
        }
        row_sync<NT, S>(rr, g);
        if (more) {
            if (!a.bulk)
                stage_x(s + nslot);
            else if (t == 0)
                stage_part(s + nslot, 1);
        }
        // ---- the round's segments in order ----
        int n = 1;   // its segments
        if constexpr (S > 1) {
            for (n = 0; n < S && s + (n - q) * R < a.K;) ++n;
        }
        float v[S][SL];
        bool ok = true;
#pragma unroll
        for (int u = 0; u < S; ++u) {
            if (u >= n) break;
            const float* from = xch + (g - q + u) * (S - 1) * SL * NT + (q < u ? q : q - 1) * SL * NT + t;
#pragma unroll
            for (int j = 0; j < SL; ++j) {
                v[u][j] = S == 1 || u == q ? own[j] : from[j * NT];
                ok = ok && is_normal(v[u][j]);
            }
        }
        if (ok) {
#pragma unroll
            for (int u = 0; u < S; ++u)
                if (u < n)
#pragma unroll
                    for (int j = 0; j < SL; ++j) acc[j] += widen(v[u][j]);
        } else {   // some zero, subnormal, infinite or undefined
#pragma unroll
            for (int u = 0; u < S; ++u)
                if (u < n)
#pragma unroll
                    for (int j = 0; j < SL; ++j) acc[j] += static_cast<double>(v[u][j]);
        }
        if (q == 0 && t == 0)
            for (int u = 0; u < n; ++u) half += static_cast<double>(halfs[g + u]);
    }
    if (row < R) {
        double* sums = a.part + row * (L + 1);
#pragma unroll
        for (int j = 0; j < SL; ++j) sums[(q * SL + j) * NT + t] = acc[j];
        if (q == 0 && t == 0) sums[L] = half;
    }
}

// Shared memory that a block of the reduction asks for and does not use: the
// blocks wait for the Welch kernel's end (dependent launch) beside its blocks,
// and without it dozens of them would crowd on one SM; so four, one a scheduler.
constexpr int kReduceSmem = 50 * 1024;

// psd[bin[i]] = scale * the sum of the rows of part in order, one thread per
// slot.  A warp's FP64 addition takes its scheduler 64 cycles, so the blocks are
// one warp each, spread over all schedulers, and the next 16 rows are requested
// before the 16 at hand are added.
__global__ void __launch_bounds__(32) psd_reduce_kernel(const double* part, int rows, int L, double scale,
                                                        const int* bin, double* psd)
{
    constexpr int kAhead = 16;
    tc::pdl_start();
    tc::pdl_wait();
    const int i = blockIdx.x * 32 + threadIdx.x;
    if (i > L) return;
    const double* p = part + i;
    const int64_t ld = L + 1;
    double s = 0.0, v[kAhead];
    int b = 0;
    if (rows >= kAhead) {
#pragma unroll
        for (int u = 0; u < kAhead; ++u) v[u] = p[u * ld];
        for (b = kAhead; b + kAhead <= rows; b += kAhead) {
            double w[kAhead];
#pragma unroll
            for (int u = 0; u < kAhead; ++u) w[u] = p[(b + u) * ld];
#pragma unroll
            for (int u = 0; u < kAhead; ++u) {
                s += v[u];
                v[u] = w[u];
            }
        }
#pragma unroll
        for (int u = 0; u < kAhead; ++u) s += v[u];
    }
#pragma unroll
    for (int u = 0; u < kAhead; ++u) v[u] = b + u < rows ? p[(b + u) * ld] : 0.0;
#pragma unroll
    for (int u = 0; u < kAhead; ++u)
        if (b + u < rows) s += v[u];
    const int k = bin[i];
    psd[k] = s * scale * ((k == 0 || k == L) ? 1.0 : 2.0);
}

// position of bin k (< L) after the in-place stages, and the tables
template <int L>
struct WelchTables {
    using W = Welch<L>;
    static int pos(int k)
    {
        const int k1 = k & 15, k2 = (k >> 4) & 15, k3 = (k >> 8) % W::R3, k4 = k / (256 * W::R3);
        return k1 * W::B + k2 * (W::B / 16) + k3 * W::R4 + k4;
    }
    static void fill(std::vector<float2>& tw, std::vector<int2>& pair0, std::vector<int>& bin)
    {
        auto root = [](int64_t m, int n) {   // W_n^m
            const double ang = -2.0 * M_PI * static_cast<double>(m) / n;
            return make_float2(static_cast<float>(std::cos(ang)), static_cast<float>(std::sin(ang)));
        };
        constexpr int R3 = W::R3, R4 = W::R4, NT = W::NT, B = W::B;
        tw.assign(W::kTables, float2{});
        for (int r = 1; r < 16; ++r)
            for (int k1 = 0; k1 < 16; ++k1) tw[W::kT2 + (r - 1) * 16 + k1] = root(r * k1 * (L / 256), L);
        for (int r = 1; r < R3; ++r)
            for (int c = 0; c < 256; ++c)
                tw[W::kT3 + (r - 1) * 256 + c] = root(r * ((c >> 4) + 16 * (c & 15)) * R4, L);
        std::vector<int> at(L);   // bin at each position
        for (int k = 0; k < L; ++k) at[pos(k)] = k;
        for (int r = 1; r < R4; ++r)
            for (int q = 0; q < L / R4; ++q) tw[W::kT4 + (r - 1) * (L / R4) + q] = root(r * at[q * R4], L);
        // a thread's 16 pairs (k, L - k): blocks k1 = 1..7 with 15..9, block 8
        // with itself, and those of block 0, whose bin L / 2 is kept apart
        pair0.clear();
        for (int k = 0; k < L / 2; k += 16) pair0.push_back(int2{zsw(pos(k)), zsw(pos((L - k) & (L - 1)))});
        bin.assign(L + 1, L / 2);
        for (int i = 0; i < 16; ++i)
            for (int t = 0; t < NT; ++t) {
                const int k1 = i < 14 ? 1 + (i >> 1) : 8, q = t + (i < 14 ? NT * (i & 1) : 0);
                const int k = i < 15 ? at[k1 * B + q] : 16 * t;
                tw[W::kSplit + i * NT + t] = root(k, W::M);
                bin[2 * i * NT + t] = k;
                bin[(2 * i + 1) * NT + t] = L - k;
            }
        tw[W::kHalf] = root(L / 2, W::M);
    }
};

struct WelchInst {
    void* fn;
    int threads, rows, smem;
    void (*fill)(std::vector<float2>&, std::vector<int2>&, std::vector<int>&);
};
template <int L>
WelchInst welch_of()
{
    return {reinterpret_cast<void*>(&psd_welch_kernel<L>), kWelchThreads, Welch<L>::ROWS, Welch<L>::kSmem,
            &WelchTables<L>::fill};
}
bool welch_inst(int L, WelchInst* w)
{
    switch (L) {
    case 2048: *w = welch_of<2048>(); return true;
    case 4096: *w = welch_of<4096>(); return true;
    case 8192: *w = welch_of<8192>(); return true;
    case 16384: *w = welch_of<16384>(); return true;
    default: return false;
    }
}

// ---------------------------------------------------------------------------
// resonance fit
// ---------------------------------------------------------------------------
constexpr int kResThreads = 256;   // threads of a block
constexpr int kResWarps = kResThreads / 32;
constexpr int kResBlocks = 8;      // blocks of the cluster
constexpr int kResRow = 32 * kResBlocks;     // points of a row: 32 per block
constexpr int kResLogRows = 64;    // rows whose ln S is kept (16,384 bins)

struct ResArgs {
    const double* psd;
    int k0, np;                // first bin and bins in the band
    double df;
    int max_iter;
    double tol, lambda0;
    double* out;               // [12]
};

// the point's contribution: the four derivatives of ln m and the residual
// (all zero, and bad set, where the model is not positive and finite)
struct ResPoint {
    double v[5];
    bool bad;
};

__device__ __forceinline__ ResPoint res_point(double f, double logS, const double (&p)[4])
{
    ResPoint o{};
    const double f0 = p[0], Q = p[1], A = p[2], B = p[3];
    const double u = f0 * f0 - f * f;
    const double c = f * f0 / Q;
    const double D = u * u + c * c;
    const double f04 = f0 * f0 * f0 * f0;
    const double g = f04 / D;
    const double m = A * g + B;
    if (!(m > 0.0) || !(m < INFINITY)) {
        o.bad = true;
        return o;
    }
    const double dD0 = 4.0 * f0 * u + 2.0 * f * f * f0 / (Q * Q);
    const double dDQ = -2.0 * c * c / Q;
    const double im = 1.0 / m;
    o.v[0] = A * (4.0 * f0 * f0 * f0 / D - f04 * dD0 / (D * D)) * im;
    o.v[1] = -A * f04 * dDQ / (D * D) * im;
    o.v[2] = g * im;
    o.v[3] = im;
    o.v[4] = logS - log(m);
    return o;
}

// (H + lambda diag H) d = g, Jacobi-scaled Cholesky; false if not positive definite
__device__ bool res_solve(const double* Hu, const double* g, double lambda, double* d)
{
    double H[4][4];
    int q = 0;
    for (int i = 0; i < 4; ++i)
        for (int j = i; j < 4; ++j) H[i][j] = H[j][i] = Hu[q++];
    double s[4];
    for (int i = 0; i < 4; ++i) {
        if (!(H[i][i] > 0.0) || !(H[i][i] < INFINITY)) return false;
        s[i] = 1.0 / sqrt(H[i][i]);
    }
    double Mx[4][4], Lc[4][4] = {};
    for (int i = 0; i < 4; ++i)
        for (int j = 0; j < 4; ++j) Mx[i][j] = (i == j) ? 1.0 + lambda : H[i][j] * s[i] * s[j];
    for (int j = 0; j < 4; ++j) {
        double v = Mx[j][j];
        for (int k = 0; k < j; ++k) v -= Lc[j][k] * Lc[j][k];
        if (!(v > 0.0)) return false;
        Lc[j][j] = sqrt(v);
        for (int i = j + 1; i < 4; ++i) {
            double w = Mx[i][j];
            for (int k = 0; k < j; ++k) w -= Lc[i][k] * Lc[j][k];
            Lc[i][j] = w / Lc[j][j];
        }
    }
    double zz[4], u[4];
    for (int i = 0; i < 4; ++i) {
        double v = g[i] * s[i];
        for (int k = 0; k < i; ++k) v -= Lc[i][k] * zz[k];
        zz[i] = v / Lc[i][i];
    }
    for (int i = 3; i >= 0; --i) {
        double v = zz[i];
        for (int k = i + 1; k < 4; ++k) v -= Lc[k][i] * u[k];
        u[i] = v / Lc[i][i];
    }
    for (int i = 0; i < 4; ++i) d[i] = u[i] * s[i];
    return true;
}

// diag(H^-1) by Gauss-Jordan with row pivoting on the 4x4 matrix (in
// registers: rows are swapped by selects); false if singular
__device__ __forceinline__ bool res_inv_diag(const double* Hu, double (&dg)[4])
{
    double A[4][8];
    int q = 0;
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = i; j < 4; ++j) A[i][j] = A[j][i] = Hu[q++];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) A[i][4 + j] = (i == j) ? 1.0 : 0.0;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        int piv = c;
        double best = fabs(A[c][c]);
#pragma unroll
        for (int r = c + 1; r < 4; ++r)
            if (fabs(A[r][c]) > best) {
                best = fabs(A[r][c]);
                piv = r;
            }
        if (!(best > 0.0)) return false;
#pragma unroll
        for (int r = c + 1; r < 4; ++r)
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const double x = A[c][j], y = A[r][j];
                A[c][j] = piv == r ? y : x;
                A[r][j] = piv == r ? x : y;
            }
        const double ip = 1.0 / A[c][c];
#pragma unroll
        for (int j = 0; j < 8; ++j) A[c][j] *= ip;
#pragma unroll
        for (int r = 0; r < 4; ++r)
            if (r != c) {
                const double fct = A[r][c];
#pragma unroll
                for (int j = 0; j < 8; ++j) A[r][j] -= fct * A[c][j];
            }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) dg[i] = A[i][4 + i];
    return true;
}

// The fit by one cluster of eight blocks.  Row c of the band (points 256 c ..)
// is split into 32 points per block; a block's warps evaluate its rows in
// parallel, then each warp adds two of the 16 sums (10 of J^T J, 4 of J^T r,
// chi^2, bad points) over the rows in order, lane by lane, and reduces the
// lanes; every block receives all blocks' sums through distributed shared
// memory, adds them in block order and takes the same step, so one cluster
// barrier per step is all that the blocks exchange.  ln S is taken once.
//
// Whether the last step is taken depends on the last bit of chi^2, so every
// operation and the order of every sum are those of the plain form, which one
// block of 256 threads would run: no reciprocal in place of a division, no
// other elimination.  What bounds it is that chain: eight divisions and a
// logarithm per point, then thirty divisions and square roots of the solve one
// after another, FP64 at 1.7 lanes a cycle and SM.  The fit of a 393-bin band
// takes 120 us (318 on one block).
__global__ void __cluster_dims__(kResBlocks, 1, 1) __launch_bounds__(kResThreads)
    resonance_fit_kernel(ResArgs a)
{
    __shared__ double red[2][kResBlocks][16];       // sums of every block, by parity of the step
    __shared__ double tot[16];
    __shared__ double pts[2][kResWarps][6][32];     // a round's points, double-buffered
    __shared__ double logs[kResLogRows][32];
    __shared__ double s_v[2][kResWarps];
    __shared__ int s_i[2][kResWarps];
    __shared__ double sp[4];        // parameters at which the sums are taken
    __shared__ int s_ctl;           // 0 continue, 1 stop
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
    const uint32_t rank = tc::cluster_rank();
    const double* S = a.psd + a.k0;
    const int rows = (a.np + kResRow - 1) / kResRow;
    tc::cluster_sync();   // every block runs before another stores into its shared memory
    tc::pdl_wait();   // (the density may come from the kernel before)
    for (int c = warp; c < rows && c < kResLogRows; c += kResWarps) {
        const int i = c * kResRow + static_cast<int>(rank) * 32 + lane;
        if (i < a.np) logs[c][lane] = log(S[i]);   // read back by this thread only
    }
    // the two sums of this warp: pairs (i, j) of J^T J row by row, then J^T r, r r and the bad points
    const int q0 = 2 * warp;
    auto pair_of = [](int q, int& i, int& j) {
        if (q < 10) {
            i = q < 4 ? 0 : q < 7 ? 1 : q < 9 ? 2 : 3;
            j = q - (i == 0 ? 0 : i == 1 ? 3 : i == 2 ? 5 : 6);
        } else {
            i = q < 14 ? q - 10 : 4;
            j = 4;
        }
    };
    int i0, j0, i1, j1;
    pair_of(q0, i0, j0);
    pair_of(q0 + 1, i1, j1);
    int parity = 0;
    // sums over the band at sp -> tot (all threads of the cluster take part)
    auto sums = [&]() {
        const double p[4] = {sp[0], sp[1], sp[2], sp[3]};
        double sa = 0.0, sb = 0.0;
        int buf = 0;
        for (int c0 = 0; c0 < rows; c0 += kResWarps, buf ^= 1) {
            const int c = c0 + warp;
            const int i = c * kResRow + static_cast<int>(rank) * 32 + lane;
            ResPoint o{};
            if (i < a.np) o = res_point((a.k0 + i) * a.df, c < kResLogRows ? logs[c][lane] : log(S[i]), p);
#pragma unroll
            for (int q = 0; q < 5; ++q) pts[buf][warp][q][lane] = o.v[q];
            pts[buf][warp][5][lane] = o.bad ? 1.0 : 0.0;
            __syncthreads();
            const int nr = rows - c0 < kResWarps ? rows - c0 : kResWarps;
            for (int k = 0; k < nr; ++k) {   // (points beyond the band add zeros)
                sa = fma(pts[buf][k][i0][lane], pts[buf][k][j0][lane], sa);
                sb = warp == kResWarps - 1 ? sb + pts[buf][k][5][lane]
                                           : fma(pts[buf][k][i1][lane], pts[buf][k][j1][lane], sb);
            }
        }
        // both sums over the lanes, distances 16, 8, 4, 2, 1: after the first
        // the lower half warp adds up the one, the upper half the other
        const bool upper = lane >= 16;
        double sum = (upper ? sb : sa) + __shfl_xor_sync(0xffffffffu, upper ? sa : sb, 16);
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
        if ((lane & 15) < kResBlocks) {   // lanes b and 16 + b hand this block's two sums to block b
            const uint32_t own = static_cast<uint32_t>(__cvta_generic_to_shared(&red[parity][rank][q0 + (upper ? 1 : 0)]));
            uint32_t there;
            asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(there) : "r"(own), "r"(lane & 15));
            asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(there), "d"(sum) : "memory");
        }
        tc::cluster_sync();
        if (t < 16) {
            double v = 0.0;
            for (int w = 0; w < kResBlocks; ++w) v += red[parity][w][t];
            tot[t] = v;
        }
        parity ^= 1;
        __syncthreads();
    };
    // initial values: the largest bin (the first of equals), the smallest
    // value, and the ends of the run above half height around the largest
    {
        double vmax = S[0], vmin = S[0];
        int kp = 0;
        for (int i = t; i < a.np; i += kResThreads) {
            const double v = S[i];
            if (v > vmax) {
                vmax = v;
                kp = i;
            }
            if (v < vmin) vmin = v;
        }
        auto merge = [&](double om, int ok, double on) {
            if (om > vmax || (om == vmax && ok < kp)) {
                vmax = om;
                kp = ok;
            }
            if (on < vmin) vmin = on;
        };
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const double om = __shfl_xor_sync(0xffffffffu, vmax, o), on = __shfl_xor_sync(0xffffffffu, vmin, o);
            merge(om, __shfl_xor_sync(0xffffffffu, kp, o), on);
        }
        if (lane == 0) {
            s_v[0][warp] = vmax;
            s_v[1][warp] = vmin;
            s_i[0][warp] = kp;
        }
        __syncthreads();
        for (int w = 0; w < kResWarps; ++w) merge(s_v[0][w], s_i[0][w], s_v[1][w]);
        const double B = vmin, h = vmax - B, half = B + 0.5 * h;
        int lo = -1, hi = a.np;   // the last bin below kp and the first above it that are not above half
        for (int i = t; i < a.np; i += kResThreads)
            if (!(S[i] > half)) {
                if (i < kp) lo = i;
                if (i > kp && i < hi) hi = i;
            }
        lo = __reduce_max_sync(0xffffffffu, lo);
        hi = __reduce_min_sync(0xffffffffu, hi);
        __syncthreads();
        if (lane == 0) {
            s_i[0][warp] = lo;
            s_i[1][warp] = hi;
        }
        __syncthreads();
        if (t == 0) {
            for (int w = 1; w < kResWarps; ++w) {
                lo = s_i[0][w] > lo ? s_i[0][w] : lo;
                hi = s_i[1][w] < hi ? s_i[1][w] : hi;
            }
            ++lo;
            --hi;
            const double fl = (lo == 0) ? (a.k0 + lo) * a.df
                                        : (a.k0 + lo - 1) * a.df + (half - S[lo - 1]) / (S[lo] - S[lo - 1]) * a.df;
            const double fh = (hi == a.np - 1) ? (a.k0 + hi) * a.df
                                               : (a.k0 + hi) * a.df + (S[hi] - half) / (S[hi] - S[hi + 1]) * a.df;
            const double width = fmax(fh - fl, a.df);
            const double f0 = (a.k0 + kp) * a.df;
            const double Q = f0 / width;
            sp[0] = f0;
            sp[1] = Q;
            sp[2] = h / (Q * Q);
            sp[3] = B;
            s_ctl = 0;
        }
        __syncthreads();
    }
    // thread 0 of each block takes the LM decisions; every block comes to the same
    double p[4], chi2 = 0.0, lambda = a.lambda0, Hc[10], gc[4];
    int it = 0, st = 1;
    bool here = true;   // the sums at hand are those at p
    sums();
    if (t == 0) {
        for (int i = 0; i < 4; ++i) p[i] = sp[i];
        chi2 = (tot[15] > 0.0) ? INFINITY : tot[14];
        for (int i = 0; i < 10; ++i) Hc[i] = tot[i];
        for (int i = 0; i < 4; ++i) gc[i] = tot[10 + i];
        if (!(chi2 < INFINITY)) {
            st = 3;
            s_ctl = 1;
        }
    }
    __syncthreads();
    while (true) {
        // the next trial point
        if (t == 0 && s_ctl == 0) {
            if (it >= a.max_iter) {
                s_ctl = 1;
            } else {
                ++it;
                double d[4];
                if (!res_solve(Hc, gc, lambda, d)) {
                    st = 2;
                    s_ctl = 1;
                } else {
                    for (int i = 0; i < 4; ++i) sp[i] = p[i] + d[i];
                }
            }
        }
        __syncthreads();
        if (s_ctl) break;
        sums();
        if (t == 0) {
            const double c2 = (tot[15] > 0.0) ? INFINITY : tot[14];
            here = false;
            if (!(c2 < INFINITY)) {
                lambda *= 10.0;
            } else if (fabs(c2 - chi2) <= a.tol * chi2) {
                if (c2 <= chi2) {
                    for (int i = 0; i < 4; ++i) p[i] = sp[i];
                    chi2 = c2;
                    here = true;
                }
                st = 0;
                s_ctl = 1;
            } else if (c2 < chi2) {
                for (int i = 0; i < 4; ++i) p[i] = sp[i];
                chi2 = c2;
                for (int i = 0; i < 10; ++i) Hc[i] = tot[i];
                for (int i = 0; i < 4; ++i) gc[i] = tot[10 + i];
                lambda *= 0.1;
                here = true;
            } else {
                lambda *= 10.0;
            }
        }
        __syncthreads();
    }
    // standard errors from the sums at the result, taken again only where the
    // last point was refused (every block of the cluster finds the same)
    __syncthreads();   // (all have read s_ctl)
    if (t == 0) {
        s_ctl = here ? 1 : 0;
        for (int i = 0; i < 4; ++i) sp[i] = p[i];
    }
    __syncthreads();
    if (!s_ctl) sums();
    if (t == 0 && rank == 0) {
        double dg[4] = {NAN, NAN, NAN, NAN};
        const bool inv = a.np > 4 && res_inv_diag(tot, dg);
        for (int i = 0; i < 4; ++i) {
            a.out[i] = sp[i];
            a.out[4 + i] = inv ? sqrt(dg[i] * chi2 / (a.np - 4)) : NAN;
        }
        a.out[8] = chi2;
        a.out[9] = it;
        a.out[10] = st;
        a.out[11] = a.np;
    }
}

}  // namespace

}  // namespace cg

using namespace cg;

namespace {
cg_status psd_fail(cg_status st, const char* msg)
{
    cg::set_last_error(msg);
    return st;
}
cg_status psd_cuda_fail(cudaError_t e, const char* what)
{
    static thread_local char buf[256];
    std::snprintf(buf, sizeof(buf), "%s: %s", what, cudaGetErrorString(e));
    cg::set_last_error(buf);
    return e == cudaErrorMemoryAllocation ? CG_ERR_NOMEM : CG_ERR_CUDA;
}
}  // namespace

cg_status cg_psd_create(int seg_len, cg_psd_t* out)
{
    if (!out) return psd_fail(CG_ERR_ARG, "out is NULL");
    *out = nullptr;
    const int L = seg_len / 2;
    WelchInst wi;
    if (seg_len % 2 != 0 || !welch_inst(L, &wi))
        return psd_fail(CG_ERR_ARG, "seg_len must be 4096, 8192, 16384 or 32768");
    cg_psd_s* h = new cg_psd_s;
    cudaGetDevice(&h->device);
    h->L = L;
    const int M = seg_len;
    std::vector<float> w(L + 1);   // w[M - n] = w[n]
    double sw2 = 0.0;
    for (int n = 0; n <= L; ++n) w[n] = static_cast<float>(0.5 - 0.5 * std::cos(2.0 * M_PI * n / M));
    for (int n = 0; n < M; ++n) {   // the window the kernel applies
        const double v = w[n <= L ? n : M - n];
        sw2 += v * v;
    }
    h->sum_w2 = sw2;
    std::vector<float2> tw;
    std::vector<int2> pair0;
    std::vector<int> bin;
    wi.fill(tw, pair0, bin);
    int sms = 0;
    cudaError_t e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, h->device);
    h->smem = wi.smem;
    h->rows = wi.rows;
    h->blocks = sms;
    auto upload = [&](auto** dst, const auto& src) {
        const size_t bytes = sizeof(src[0]) * src.size();
        if (e == cudaSuccess) e = cudaMalloc(dst, bytes);
        if (e == cudaSuccess) e = cudaMemcpy(*dst, src.data(), bytes, cudaMemcpyHostToDevice);
    };
    if (e == cudaSuccess) e = cg::raise_smem_limit(wi.fn, wi.smem);
    if (e == cudaSuccess) e = cg::raise_smem_limit(reinterpret_cast<void*>(&psd_reduce_kernel), kReduceSmem);
    upload(&h->win, w);
    upload(&h->tw, tw);
    upload(&h->pair0, pair0);
    upload(&h->bin, bin);
    if (e == cudaSuccess)
        e = cudaMalloc(&h->part, sizeof(double) * (L + 1) * static_cast<size_t>(h->blocks) * h->rows);
    if (e != cudaSuccess) {
        cg_psd_destroy(h);
        return psd_cuda_fail(e, "cg_psd_create");
    }
    *out = h;
    return CG_OK;
}

void cg_psd_destroy(cg_psd_t h)
{
    if (!h) return;
    cudaFree(h->win);
    cudaFree(h->tw);
    cudaFree(h->pair0);
    cudaFree(h->bin);
    cudaFree(h->part);
    delete h;
}

cg_status cg_psd_welch(cg_psd_t h, const float* x_dev, int64_t n, int64_t stride, double fs, double* psd_dev,
                       int64_t* n_segments, void* stream)
{
    if (!h || !x_dev || !psd_dev) return psd_fail(CG_ERR_ARG, "handle, x_dev and psd_dev are required");
    if (stride < 1) return psd_fail(CG_ERR_ARG, "stride must be >= 1");
    if (!(fs > 0.0) || !std::isfinite(fs)) return psd_fail(CG_ERR_ARG, "fs must be > 0");
    const int64_t M = 2LL * h->L;
    if (n < M) return psd_fail(CG_ERR_ARG, "series shorter than one segment");
    const int64_t K = (n - M) / h->L + 1;
    if (n_segments) *n_segments = K;
    const cudaStream_t s = static_cast<cudaStream_t>(stream);
    const int vec2 = stride == 1 && (reinterpret_cast<uintptr_t>(x_dev) & 7) == 0;
    const int bulk = stride == 1 && (reinterpret_cast<uintptr_t>(x_dev) & 15) == 0;
    // the rows go to different SMs before they share one
    const int rows = static_cast<int>(std::min<int64_t>(K, static_cast<int64_t>(h->blocks) * h->rows));
    const int grid = std::min(rows, h->blocks);
    PsdArgs a{x_dev, stride, K, rows, vec2, bulk, h->win, h->tw, h->pair0, h->part};
    WelchInst wi;
    welch_inst(h->L, &wi);
    void* args[] = {&a};
    cudaError_t e = cudaLaunchKernel(wi.fn, dim3(grid), dim3(wi.threads), args, h->smem, s);
    if (e == cudaSuccess) {
        const double scale = 1.0 / (static_cast<double>(K) * fs * h->sum_w2);
        const double* part = h->part;
        const int* bin = h->bin;
        void* rargs[] = {&part, const_cast<int*>(&rows), &h->L, const_cast<double*>(&scale), &bin, &psd_dev};
        e = launch_dependent(reinterpret_cast<void*>(&psd_reduce_kernel), dim3((h->L + 1 + 31) / 32), dim3(32), rargs,
                             kReduceSmem, s);
    }
    if (e != cudaSuccess) return psd_cuda_fail(e, "cg_psd_welch");
    return CG_OK;
}

cg_status cg_resonance_fit(const double* psd_dev, int n_bins, double df, double f_lo, double f_hi, int max_iter,
                           double tol, double* out_dev, void* stream)
{
    if (!psd_dev || !out_dev) return psd_fail(CG_ERR_ARG, "psd_dev and out_dev are required");
    if (n_bins < 8 || !(df > 0.0) || !(f_hi > f_lo) || max_iter < 0 || !(tol >= 0.0))
        return psd_fail(CG_ERR_ARG, "need n_bins >= 8, df > 0, f_hi > f_lo, max_iter >= 0, tol >= 0");
    int k0 = static_cast<int>(std::ceil(f_lo / df));
    int k1 = static_cast<int>(std::floor(f_hi / df));
    if (k0 < 1) k0 = 1;                       // the model's f = 0 point carries no resonance information
    if (k1 > n_bins - 1) k1 = n_bins - 1;
    if (k1 - k0 + 1 < 8) return psd_fail(CG_ERR_ARG, "the band holds fewer than 8 bins");
    ResArgs a{psd_dev, k0, k1 - k0 + 1, df, max_iter, tol, 1e-3, out_dev};
    void* args[] = {&a};
    cudaError_t e = launch_dependent(reinterpret_cast<void*>(&resonance_fit_kernel), dim3(kResBlocks),
                                     dim3(kResThreads), args, 0, static_cast<cudaStream_t>(stream));
    if (e != cudaSuccess) return psd_cuda_fail(e, "cg_resonance_fit");
    return CG_OK;
}
