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
// over all their segments as FP32 pairs; the groups' rows are summed and
// scaled by psd_reduce_kernel.
//
// Resonance: S(f) = A f0^4 / ((f0^2 - f^2)^2 + (f f0 / Q)^2) + B fitted to
// ln S over the bins of a band by Levenberg-Marquardt in FP64 (one block:
// per-point sums reduced in shared memory, the 4x4 solve on one thread);
// initial values from the band (largest bin, smallest bin, half-height
// width); standard errors from diag(H^-1) chi^2 / (n - 4).
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <vector>
#include <cuda_runtime.h>

#include "cg_fft.cuh"
#include "cg_internal.h"
#include "cg_stage.cuh"

namespace cg {
constexpr int kWelchThreads = 512;   // threads of a block of the Welch kernel
}

struct cg_psd_s {
    int device = 0;
    int L = 0;                 // complex transform length (M / 2)
    int grid = 0;              // blocks of the Welch kernel at most
    int groups = 0;            // segments a block transforms at a time
    size_t smem = 0;
    double sum_w2 = 0.0;       // sum of the squared window
    float* win = nullptr;      // [M / 2 + 1] the window's first half (it is symmetric)
    float2* tw = nullptr;      // the kernel's twiddles (WelchTables)
    int2* pair0 = nullptr;     // [L / 32] buffer places of the last pair of each thread
    int* bin = nullptr;        // [L + 1] PSD bin of each slot of a row of part
    float2* part = nullptr;    // [grid * groups][L + 1] sums of |X_k|^2 as FP32 pairs
};

namespace cg {

namespace {

// The transform of one segment: L = 16 * 16 * R3 * R4 complex points, by a
// group of L / 32 threads (each 32 points).
template <int L>
struct Welch {
    static constexpr int NT = L / 32;                   // threads of a group
    static constexpr int G = kWelchThreads / NT;        // groups of a block
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
    // the window, warp sums, the extra bin's sum of each group
    static constexpr int kSmemZ = G * L * 8;
    static constexpr int kSmemT = kSmemZ + (15 * 16 + (R3 - 1) * 256) * 8;
    static constexpr int kSmemW = kSmemT + (M / 2 + 4) * 4;
    static constexpr int kSmem = kSmemW + G * (2 * NT / 32) * 4 + G * 8;
};

struct PsdArgs {
    const float* x;
    int64_t stride;            // elements between consecutive samples
    int64_t K;                 // segments
    int vec2;                  // sample pairs are 8-byte aligned and contiguous
    const float* win;
    const float2* tw;
    const int2* pair0;
    float2* part;
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

// s + e = a + b exactly (Knuth's two-sum)
__device__ __forceinline__ float two_sum(float a, float b, float& e)
{
    const float s = a + b, bb = s - a;
    e = (a - (s - bb)) + (b - bb);
    return s;
}

// Sums of |X_k|^2 as unevaluated FP32 pairs (hi, lo).  An FP64 sum costs a
// conversion and an addition at 2 lanes per cycle and SM (16,384 bins: 16,000
// cycles of a segment's 61,000); the pair costs 7 FP32 operations at 128 lanes
// per cycle.  The lost part of each addition is exact; lo, kept below an ulp
// of hi by a normalisation every eighth segment, rounds it 2^-24 below that.
__device__ __forceinline__ void pair_add(float2& a, float b)
{
    float e;
    a.x = two_sum(a.x, b, e);
    a.y += e;
}
// an infinite or undefined sum stays what it is
__device__ __forceinline__ void pair_norm(float2& a)
{
    const float h = a.x + a.y;
    const bool fin = fabsf(a.x) < INFINITY;
    a = make_float2(fin ? h : a.x, fin ? a.y - (h - a.x) : 0.f);
}
__device__ __forceinline__ void pair_add2(float2& a, float2 b)
{
    pair_add(a, b.x);
    a.y += b.y;
    pair_norm(a);
}

// Welch sums.  One segment per group of NT threads, its L packed complex
// values z_n = x_2n + i x_2n+1 in shared memory.  The transform runs in place
// (digit-reversed result): the points of a butterfly go back where they were
// read, so a thread needs no barrier between its reads and its writes, and
// after the first stage (stride L / 16) all remaining butterflies of a warp
// stay inside the warp's own 1,024 points -- two block barriers per
// transform instead of eight, and 16 live values per thread.  That leaves the
// registers for the sums of |X_k|^2: the thread that holds bins k and L - k
// (one split, two bins from the same two points and twiddle) adds them up over
// all its segments.
//
// What bounds it: shared-memory traffic (1.3 MB per 32,768-sample segment,
// 10,000 cycles) and the transform's FP32 work.  Before, the sums lived in
// L2 as FP64 rows and every table but one was read from L2 (0.75 MB per
// segment), the sums and the mean ran in FP64 on every thread, and each stage
// took two barriers of 1,024 threads.  Ten minutes of centres (36,620
// segments of 32,768): 7.99 -> 3.11 ms (27,000 cycles a segment; the shared
// memory is busy for 54 % of them).
template <int L>
__global__ void __launch_bounds__(kWelchThreads, 1) psd_welch_kernel(PsdArgs a)
{
    using W = Welch<L>;
    constexpr int NT = W::NT, R3 = W::R3, R4 = W::R4, B = W::B, M = W::M, G = W::G;
    extern __shared__ __align__(1024) unsigned char psm[];
    const int g = threadIdx.x / NT, t = threadIdx.x % NT, w = t >> 5, lane = t & 31;
    const uint32_t z = static_cast<uint32_t>(__cvta_generic_to_shared(psm)) + g * L * 8;
    float2* const ts = reinterpret_cast<float2*>(psm + W::kSmemZ);
    const float2* const t2 = ts + W::kT2;
    const float2* const t3 = ts + W::kT3;
    float* const win = reinterpret_cast<float*>(psm + W::kSmemT);
    float* const red = reinterpret_cast<float*>(psm + W::kSmemW) + g * (2 * NT / 32);
    float2* const half = reinterpret_cast<float2*>(psm + W::kSmemW + G * (2 * NT / 32) * 4) + g;
    const int64_t slot = static_cast<int64_t>(g) * gridDim.x + blockIdx.x;   // this group's first segment
    const int64_t nslot = static_cast<int64_t>(G) * gridDim.x;
    const uint32_t zt = z + 8 * zsw(t);             // point t, and NT - 1 - t
    const uint32_t zr = z + 8 * zsw(NT - 1 - t);

    auto stage_x = [&](int64_t s) {   // the thread's own 32 points of segment s, asynchronously
        const float* x = a.x + s * static_cast<int64_t>(L) * a.stride;
        if (a.vec2) {
            x += 2 * t;
#pragma unroll 8
            for (int i = 0; i < 32; ++i)
                asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(zat(zt, NT * i)), "l"(x + 2 * NT * i) : "memory");
        } else {
            x += 2 * t * a.stride;
#pragma unroll 4
            for (int i = 0; i < 32; ++i) {
                const float* p = x + 2 * NT * i * a.stride;
                asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(zat(zt, NT * i)), "l"(p) : "memory");
                asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(zat(zt, NT * i) + 4), "l"(p + a.stride) : "memory");
            }
        }
        cp_async_commit();
    };
    if (slot < a.K) stage_x(slot);
    for (int i = threadIdx.x; i < W::kT4; i += kWelchThreads) ts[i] = a.tw[i];
    for (int i = threadIdx.x; i <= M / 2; i += kWelchThreads) win[i] = a.win[i];
    if (t == 0) *half = make_float2(0.f, 0.f);
    const int2 p15 = a.pair0[t];
    float2 acc[16][2];
#pragma unroll
    for (int i = 0; i < 16; ++i) acc[i][0] = acc[i][1] = make_float2(0.f, 0.f);
    __syncthreads();

    int since = 0;   // segments since the sums were normalised
    for (int64_t s = slot; s < a.K; s += nslot) {
        // the next segment into L2 meanwhile
        if (s + nslot < a.K && a.stride <= 4) {
            const char* nx = reinterpret_cast<const char*>(a.x + (s + nslot) * static_cast<int64_t>(L) * a.stride);
            for (int64_t i = t; i < M * a.stride / 32; i += NT) asm volatile("prefetch.global.L2 [%0];\n" ::"l"(nx + 128 * i));
        }
        cp_async_wait_all();   // own points only: no barrier
        // ---- segment mean: FP32 sums of 32 samples per first-stage column ----
#pragma unroll
        for (int b = 0; b < 2; ++b) {
            float sum = 0.0f;
#pragma unroll
            for (int r = 0; r < 16; ++r) {
                const float2 v = zld(zat(zt, NT * (b + 2 * r)));
                sum += v.x + v.y;
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
            if (lane == 0) red[w + (NT / 32) * b] = sum;
        }
        group_sync<NT>(g);
        // every warp adds the warp sums as FP32 pairs (48 bits) and rounds once
        float2 tot = make_float2(lane < 2 * NT / 32 ? red[lane] : 0.f, 0.f);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
            pair_add2(tot, make_float2(__shfl_xor_sync(0xffffffffu, tot.x, o), __shfl_xor_sync(0xffffffffu, tot.y, o)));
        const float mean = tot.x * (1.0f / M);
        // ---- stage 1: subtract the mean, window, 16 points at stride B ----
#pragma unroll 1
        for (int b = 0; b < 2; ++b) {
            const int j = t + NT * b;
            const uint32_t zj = zat(zt, NT) * b + zt * (1 - b);
            float2 v[16];
#pragma unroll
            for (int r = 0; r < 16; ++r) {
                const int n = j + r * B;
                v[r] = zld(zat(zj, r * B));
                float2 wn;
                if (r < 8)
                    wn = *reinterpret_cast<const float2*>(win + 2 * n);
                else
                    wn = make_float2(win[M - 2 * n], win[M - 2 * n - 1]);
                v[r] = make_float2((v[r].x - mean) * wn.x, (v[r].y - mean) * wn.y);
            }
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
#pragma unroll 4
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
        group_sync<NT>(g);
        // ---- real-FFT split of bins k and L - k, |X|^2 into the sums ----
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            const int k1 = i < 14 ? 1 + (i >> 1) : 8, h = i < 14 ? i & 1 : 0;
            const float2 Zb = zld(i < 15 ? zat(zt, k1 * B + NT * h) : z + 8 * p15.x);
            const float2 Zr = zld(i < 15 ? zat(zr, (16 - k1) * B + NT * (1 - h)) : z + 8 * p15.y);
            const float2 E = make_float2(0.5f * (Zb.x + Zr.x), 0.5f * (Zb.y - Zr.y));
            const float2 Dd = make_float2(0.5f * (Zb.x - Zr.x), 0.5f * (Zb.y + Zr.y));
            const float2 C = cmul(__ldg(&a.tw[W::kSplit + i * NT + t]), make_float2(Dd.y, -Dd.x));
            // X_k = E + C; X_(L - k) = conj(E - C), since W_M^(L - k) = -conj W_M^k
            const float2 X = cadd(E, C), Y = csub(E, C);
            pair_add(acc[i][0], fmaf(X.x, X.x, X.y * X.y));
            pair_add(acc[i][1], fmaf(Y.x, Y.x, Y.y * Y.y));
        }
        if (t == 0) {   // bin L / 2 pairs with itself
            constexpr int kPos = R4 > 1 ? R4 / 2 : R3 / 2;   // its last digit is R / 2, the others 0
            const float2 Zh = zld(z + 8 * zsw(kPos));
            const float2 X = cadd(make_float2(Zh.x, 0.f), cmul(__ldg(&a.tw[W::kHalf]), make_float2(Zh.y, -0.f)));
            pair_add2(*half, make_float2(fmaf(X.x, X.x, X.y * X.y), 0.f));
        }
        group_sync<NT>(g);
        if (s + nslot < a.K) stage_x(s + nslot);
        if (++since == 8 || s + nslot >= a.K) {
            since = 0;
#pragma unroll
            for (int i = 0; i < 16; ++i) {
                pair_norm(acc[i][0]);
                pair_norm(acc[i][1]);
            }
        }
    }
    if (slot < a.K) {
        float2* row = a.part + slot * (L + 1);
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            row[(2 * i) * NT + t] = acc[i][0];
            row[(2 * i + 1) * NT + t] = acc[i][1];
        }
        if (t == 0) row[L] = *half;
    }
}

// psd[bin[i]] = scale * sum over the rows of part: 32 slots per block, eight
// threads per slot over rows y, y + 8, ..., then in order of y (fixed order).
// The rows are summed as FP32 pairs too: 152 rows of 16,385 bins took 22 us as
// FP64 additions on 65 blocks, 8 us so (60 rows: 10.9 and 5.6 us).
__global__ void __launch_bounds__(256) psd_reduce_kernel(const float2* part, int rows, int L, double scale,
                                                         const int* bin, double* psd)
{
    __shared__ float2 red[8][33];
    const int i = blockIdx.x * 32 + threadIdx.x;
    float2 s = make_float2(0.f, 0.f);
    if (i <= L) {
#pragma unroll 4
        for (int b = threadIdx.y; b < rows; b += 8) {
            const float2 v = part[static_cast<int64_t>(b) * (L + 1) + i];
            pair_add2(s, v);
        }
    }
    red[threadIdx.y][threadIdx.x] = s;
    __syncthreads();
    if (threadIdx.y == 0 && i <= L) {
        for (int y = 1; y < 8; ++y) pair_add2(s, red[y][threadIdx.x]);
        const int k = bin[i];
        psd[k] = (static_cast<double>(s.x) + static_cast<double>(s.y)) * scale * ((k == 0 || k == L) ? 1.0 : 2.0);
    }
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
    int threads, groups, smem;
    void (*fill)(std::vector<float2>&, std::vector<int2>&, std::vector<int>&);
};
template <int L>
WelchInst welch_of()
{
    return {reinterpret_cast<void*>(&psd_welch_kernel<L>), kWelchThreads, Welch<L>::G, Welch<L>::kSmem,
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
constexpr int kResThreads = 256;

struct ResArgs {
    const double* psd;
    int k0, np;                // first bin and bins in the band
    double df;
    int max_iter;
    double tol, lambda0;
    double* out;               // [12]
};

// per-point sums: 10 of J^T J (upper), 4 of J^T r, chi^2, bad-point count
struct ResSums {
    double v[16];
};

__device__ __forceinline__ void res_point(double f, double S, const double (&p)[4], ResSums& s)
{
    const double f0 = p[0], Q = p[1], A = p[2], B = p[3];
    const double u = f0 * f0 - f * f;
    const double c = f * f0 / Q;
    const double D = u * u + c * c;
    const double f04 = f0 * f0 * f0 * f0;
    const double g = f04 / D;
    const double m = A * g + B;
    if (!(m > 0.0) || !(m < INFINITY)) {
        s.v[15] += 1.0;
        return;
    }
    const double dD0 = 4.0 * f0 * u + 2.0 * f * f * f0 / (Q * Q);
    const double dDQ = -2.0 * c * c / Q;
    const double im = 1.0 / m;
    double J[4];
    J[0] = A * (4.0 * f0 * f0 * f0 / D - f04 * dD0 / (D * D)) * im;
    J[1] = -A * f04 * dDQ / (D * D) * im;
    J[2] = g * im;
    J[3] = im;
    const double r = log(S) - log(m);
    int q = 0;
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = i; j < 4; ++j) s.v[q++] += J[i] * J[j];
#pragma unroll
    for (int i = 0; i < 4; ++i) s.v[10 + i] += J[i] * r;
    s.v[14] += r * r;
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

// diag(H^-1) by Gauss-Jordan on the 4x4 matrix; false if singular
__device__ bool res_inv_diag(const double* Hu, double* dg)
{
    double A[4][8];
    int q = 0;
    for (int i = 0; i < 4; ++i)
        for (int j = i; j < 4; ++j) A[i][j] = A[j][i] = Hu[q++];
    for (int i = 0; i < 4; ++i)
        for (int j = 0; j < 4; ++j) A[i][4 + j] = (i == j) ? 1.0 : 0.0;
    for (int c = 0; c < 4; ++c) {
        int piv = c;
        for (int r = c + 1; r < 4; ++r)
            if (fabs(A[r][c]) > fabs(A[piv][c])) piv = r;
        if (!(fabs(A[piv][c]) > 0.0)) return false;
        for (int j = 0; j < 8; ++j) {
            const double tmp = A[c][j];
            A[c][j] = A[piv][j];
            A[piv][j] = tmp;
        }
        const double ip = 1.0 / A[c][c];
        for (int j = 0; j < 8; ++j) A[c][j] *= ip;
        for (int r = 0; r < 4; ++r)
            if (r != c) {
                const double fct = A[r][c];
                for (int j = 0; j < 8; ++j) A[r][j] -= fct * A[c][j];
            }
    }
    for (int i = 0; i < 4; ++i) dg[i] = A[i][4 + i];
    return true;
}

__global__ void __launch_bounds__(kResThreads) resonance_fit_kernel(ResArgs a)
{
    __shared__ double red[kResThreads / 32][16];
    __shared__ ResSums tot;
    __shared__ double sp[4];        // parameters at which the sums are taken
    __shared__ int s_ctl;           // 0 continue, 1 stop
    const int t = threadIdx.x;
    const double* S = a.psd + a.k0;
    // sums over the band at sp -> tot (all threads take part)
    auto sums = [&]() {
        ResSums s;
#pragma unroll
        for (int i = 0; i < 16; ++i) s.v[i] = 0.0;
        const double p[4] = {sp[0], sp[1], sp[2], sp[3]};
        for (int i = t; i < a.np; i += kResThreads) res_point((a.k0 + i) * a.df, S[i], p, s);
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            double v = s.v[i];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
            if ((t & 31) == 0) red[t >> 5][i] = v;
        }
        __syncthreads();
        if (t < 16) {
            double v = 0.0;
            for (int w = 0; w < kResThreads / 32; ++w) v += red[w][t];
            tot.v[t] = v;
        }
        __syncthreads();
    };
    // initial values (one thread, a pass over the band)
    if (t == 0) {
        int kp = 0;
        double B = S[0];
        for (int i = 1; i < a.np; ++i) {
            if (S[i] > S[kp]) kp = i;
            if (S[i] < B) B = S[i];
        }
        const double h = S[kp] - B, half = B + 0.5 * h;
        int lo = kp, hi = kp;
        while (lo > 0 && S[lo - 1] > half) --lo;
        while (hi < a.np - 1 && S[hi + 1] > half) ++hi;
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
    double p[4], chi2 = 0.0, lambda = a.lambda0, Hc[10], gc[4];
    int it = 0, st = 1;
    sums();
    if (t == 0) {
        for (int i = 0; i < 4; ++i) p[i] = sp[i];
        chi2 = (tot.v[15] > 0.0) ? INFINITY : tot.v[14];
        for (int i = 0; i < 10; ++i) Hc[i] = tot.v[i];
        for (int i = 0; i < 4; ++i) gc[i] = tot.v[10 + i];
        if (!(chi2 < INFINITY)) {
            st = 3;
            s_ctl = 1;
        }
    }
    __syncthreads();
    while (true) {
        // thread 0 proposes a trial point
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
            const double c2 = (tot.v[15] > 0.0) ? INFINITY : tot.v[14];
            if (!(c2 < INFINITY)) {
                lambda *= 10.0;
            } else if (fabs(c2 - chi2) <= a.tol * chi2) {
                if (c2 <= chi2) {
                    for (int i = 0; i < 4; ++i) p[i] = sp[i];
                    chi2 = c2;
                }
                st = 0;
                s_ctl = 1;
            } else if (c2 < chi2) {
                for (int i = 0; i < 4; ++i) p[i] = sp[i];
                chi2 = c2;
                for (int i = 0; i < 10; ++i) Hc[i] = tot.v[i];
                for (int i = 0; i < 4; ++i) gc[i] = tot.v[10 + i];
                lambda *= 0.1;
            } else {
                lambda *= 10.0;
            }
        }
        __syncthreads();
    }
    // standard errors from the sums at the result
    if (t == 0)
        for (int i = 0; i < 4; ++i) sp[i] = p[i];
    __syncthreads();
    sums();
    if (t == 0) {
        double dg[4] = {NAN, NAN, NAN, NAN};
        const bool inv = a.np > 4 && res_inv_diag(tot.v, dg);
        for (int i = 0; i < 4; ++i) {
            a.out[i] = p[i];
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
    h->groups = wi.groups;
    h->grid = sms;
    auto upload = [&](auto** dst, const auto& src) {
        const size_t bytes = sizeof(src[0]) * src.size();
        if (e == cudaSuccess) e = cudaMalloc(dst, bytes);
        if (e == cudaSuccess) e = cudaMemcpy(*dst, src.data(), bytes, cudaMemcpyHostToDevice);
    };
    if (e == cudaSuccess) e = cg::raise_smem_limit(wi.fn, wi.smem);
    upload(&h->win, w);
    upload(&h->tw, tw);
    upload(&h->pair0, pair0);
    upload(&h->bin, bin);
    if (e == cudaSuccess)
        e = cudaMalloc(&h->part, sizeof(float2) * (L + 1) * static_cast<size_t>(h->grid) * h->groups);
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
    PsdArgs a{x_dev, stride, K, vec2, h->win, h->tw, h->pair0, h->part};
    WelchInst wi;
    welch_inst(h->L, &wi);
    // one block per SM; the segments go to different SMs before they share one
    const int grid = static_cast<int>(K < h->grid ? K : h->grid);
    const int64_t slots = static_cast<int64_t>(grid) * h->groups;
    const int rows = static_cast<int>(K < slots ? K : slots);
    void* args[] = {&a};
    cudaError_t e = cudaLaunchKernel(wi.fn, dim3(grid), dim3(wi.threads), args, h->smem, s);
    if (e == cudaSuccess) {
        const double scale = 1.0 / (static_cast<double>(K) * fs * h->sum_w2);
        psd_reduce_kernel<<<(h->L + 1 + 31) / 32, dim3(32, 8), 0, s>>>(h->part, rows, h->L, scale, h->bin, psd_dev);
        e = cudaGetLastError();
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
    cudaError_t e = cudaLaunchKernel(reinterpret_cast<void*>(&resonance_fit_kernel), dim3(1), dim3(kResThreads),
                                     args, 0, static_cast<cudaStream_t>(stream));
    if (e != cudaSuccess) return psd_cuda_fail(e, "cg_resonance_fit");
    return CG_OK;
}
