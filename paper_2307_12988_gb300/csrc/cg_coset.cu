// cg_coset.cu -- the tooth readout of comb geometries whose tooth bins lie in
// one residue pair +-r mod 10 (every 1 us-frame workload: N = 10 L, L = 10 Q).
//
// Paper ("Data Capture and Processing"): cast on the GPU, FFT per row, tooth
// bins selected and mapped, reference normalisation.  Only X at the bins
// 10 q + r is needed: with n = m + L j (m < L, j < 10)
//     X_{10 q + r} = sum_m W_L^{q m} z_m,  z_m = W_N^{r m} sum_j x_{m + L j} W_10^{r j},
// a fold to L values and an L-point transform, m = a + 10 b, q = u + Q v:
//   stage A  fold of the samples at m and, over b, the Q-point transform
//            (Q = 10, 11), or its first factor R1 (Q = R1 R2 = 22, 25);
//   stage B  (Q = 22, 25) its second factor R2;
//   stage C  the 10-point transform over a, |X|, and the two stores per tooth.
//
// What bounds it: HBM (2 N + 8 T bytes per frame) where the issue slots and
// the shared-memory port allow, so the layout saves both:
//  * samples are read two at a time (a = 2 p and 2 p + 1), and stages A and B
//    run both residues' transforms in the halves of packed FP32x2 operations;
//  * a sample becomes a float by one byte permutation: the bits of 2^23 + (x +
//    bias).  Sums and differences of those are exact, as integers were;
//  * the two 5-point transforms of stage C are the halves of another pair;
//  * every stage's items fill the block's threads (5 Q/R1 .. 5 R2 per frame in
//    A, 5 R1 in B, Q in C), and a value keeps its place between the stages;
//  * a batch's samples arrive by one bulk copy, issued when stage A has read
//    the batch before; tooth number and 1 / reference share one table entry.
// 10^6 frames of 1,100 samples take 439 us, 10^5 of 2,500 samples 111, 250,000 of
// 2,200 8-bit samples 207 (560 warp instructions and 150 shared-memory
// wavefronts per frame, 16 warps per SM); single transforms fed by 16-bit loads,
// integer folds and 16-byte cp.async took 566, 165 and 256.  At the rate of a
// copy, half of whose bytes are writes, their bytes would take 441, 100 and 111:
// no upper bound for these kernels, three quarters of whose bytes are reads.
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cuda_runtime.h>

#include "cg_fft.cuh"
#include "cg_internal.h"
#include "cg_tc.cuh"

namespace cg {

namespace {

constexpr int kP = 10;        // points of the last stage
constexpr int kHalf = kP / 2; // residue pairs

template <int R>
__device__ const RootTable<R> kRoots{};   // cos, sin of 2 pi j / R

// complex values of two transforms, one in each half
struct C2 {
    float2 re, im;
};

__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __ffma2_rn(b, make_float2(-1.f, -1.f), a); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 neg2(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ float2 dup2(float v) { return make_float2(v, v); }

// a (t.re + i t.im), rounded as cmul
__device__ __forceinline__ C2 cmul2(C2 a, float2 tr, float2 ti)
{
    return {fma2(a.re, tr, neg2(mul2(a.im, ti))), fma2(a.re, ti, mul2(a.im, tr))};
}
// a (c - i s), rounded as in DftComposite
__device__ __forceinline__ C2 crot2(C2 a, float2 c, float2 s)
{
    return {fma2(a.re, c, mul2(a.im, s)), fma2(a.im, c, neg2(mul2(a.re, s)))};
}

// the transforms of cg_fft.cuh on pairs: the same operations in the same order
template <int R>
struct PairDft {   // odd R (DftOdd)
    static __device__ __forceinline__ void run(C2 (&a)[R])
    {
        constexpr int H = (R - 1) / 2;
        constexpr RootTable<R> tab{};
        C2 s[H + 1], d[H + 1];
#pragma unroll
        for (int t = 1; t <= H; ++t) {
            s[t] = {add2(a[t].re, a[R - t].re), add2(a[t].im, a[R - t].im)};
            d[t] = {sub2(a[t].re, a[R - t].re), sub2(a[t].im, a[R - t].im)};
        }
        const C2 a0 = a[0];
#pragma unroll
        for (int t = 1; t <= H; ++t) a[0] = {add2(a[0].re, s[t].re), add2(a[0].im, s[t].im)};
#pragma unroll
        for (int v = 1; v <= H; ++v) {
            C2 P = a0, Q = {dup2(0.f), dup2(0.f)};
#pragma unroll
            for (int t = 1; t <= H; ++t) {
                const float2 c = dup2(tab.c[(v * t) % R]), sn = dup2(tab.s[(v * t) % R]);
                P = {fma2(s[t].re, c, P.re), fma2(s[t].im, c, P.im)};
                Q = {fma2(d[t].re, sn, Q.re), fma2(d[t].im, sn, Q.im)};
            }
            a[v] = {add2(P.re, Q.im), sub2(P.im, Q.re)};
            a[R - v] = {sub2(P.re, Q.im), add2(P.im, Q.re)};
        }
    }
};
template <>
struct PairDft<2> {
    static __device__ __forceinline__ void run(C2 (&a)[2])
    {
        const C2 t = a[1];
        a[1] = {sub2(a[0].re, t.re), sub2(a[0].im, t.im)};
        a[0] = {add2(a[0].re, t.re), add2(a[0].im, t.im)};
    }
};
template <>
struct PairDft<10> {   // DftComposite<2, 5>
    static __device__ __forceinline__ void run(C2 (&a)[10])
    {
        constexpr RootTable<10> tab{};
        C2 b[2][5];
#pragma unroll
        for (int n = 0; n < 5; ++n) {
            C2 v[2] = {a[n], a[5 + n]};
            PairDft<2>::run(v);
            b[0][n] = v[0];
            b[1][n] = n ? crot2(v[1], dup2(tab.c[n]), dup2(tab.s[n])) : v[1];
        }
#pragma unroll
        for (int k1 = 0; k1 < 2; ++k1) {
            PairDft<5>::run(b[k1]);
#pragma unroll
            for (int k2 = 0; k2 < 5; ++k2) a[k1 + 2 * k2] = b[k1][k2];
        }
    }
};

// Two neighbouring samples, each offset by half its range so that its bytes
// are those of an unsigned value, as 2^23 + that value.
template <class S, bool EVEN>
__device__ __forceinline__ float2 sample_pair(const S* p)
{
    if constexpr (sizeof(S) == 2) {
        const uint32_t w = *reinterpret_cast<const uint32_t*>(p) ^ 0x80008000u;
        return make_float2(__uint_as_float(__byte_perm(w, 0x4B000000u, 0x7610)),
                           __uint_as_float(__byte_perm(w, 0x4B000000u, 0x7632)));
    } else {
        uint32_t w;
        if constexpr (EVEN)
            w = *reinterpret_cast<const uint16_t*>(p);
        else   // samples at an odd address
            w = static_cast<uint32_t>(static_cast<uint8_t>(p[0])) | (static_cast<uint32_t>(static_cast<uint8_t>(p[1])) << 8);
        w ^= 0x8080u;
        return make_float2(__uint_as_float(__byte_perm(w, 0x4B000000u, 0x7640)),
                           __uint_as_float(__byte_perm(w, 0x4B000000u, 0x7641)));
    }
}

// z_m for m and m + 1 from the samples at m + L j.  With s = (-1)^r,
// w_{5-j} = s conj(w_j) for w_j = W_10^{r j}, so sum_j D_j w_j = D_0 +
// (E_1 c_1 + E_2 c_2) + i (F_1 s_1 + F_2 s_2) where D_j = x_j + s x_{j+5},
// E_j = D_j + s D_{5-j}, F_j = D_j - s D_{5-j}.
template <int L, class S, int SG, bool EVEN>
__device__ __forceinline__ C2 fold_pair(const S* x, float4 tw, float c1, float s1, float c2, float s2)
{
    constexpr float kTwice = 2.0f * (8388608.0f + (sizeof(S) == 2 ? 32768.0f : 128.0f));
    float2 D[5];
#pragma unroll
    for (int j = 0; j < 5; ++j) {
        const float2 a = sample_pair<S, EVEN>(x + L * j), b = sample_pair<S, EVEN>(x + L * (j + 5));
        if constexpr (SG < 0)
            D[j] = sub2(a, b);                                // the offsets cancel
        else
            D[j] = add2(a, add2(b, dup2(-kTwice)));           // b - 2 offset: an integer below 2^24
    }
    const float2 E1 = SG < 0 ? sub2(D[1], D[4]) : add2(D[1], D[4]), F1 = SG < 0 ? add2(D[1], D[4]) : sub2(D[1], D[4]);
    const float2 E2 = SG < 0 ? sub2(D[2], D[3]) : add2(D[2], D[3]), F2 = SG < 0 ? add2(D[2], D[3]) : sub2(D[2], D[3]);
    C2 z;
    z.re = fma2(E2, dup2(c2), fma2(E1, dup2(c1), D[0]));
    z.im = fma2(F2, dup2(s2), mul2(F1, dup2(s1)));
    return cmul2(z, make_float2(tw.x, tw.y), make_float2(tw.z, tw.w));
}

__device__ __forceinline__ C2 unpack(float4 v) { return {make_float2(v.x, v.y), make_float2(v.z, v.w)}; }
__device__ __forceinline__ float4 pack(C2 z) { return make_float4(z.re.x, z.re.y, z.im.x, z.im.y); }

// float4 entries per frame between the stages: 5 Q, and 5 mod 8 so that items
// of neighbouring frames go on where the frame's own end in the banks
template <int Q>
constexpr int frame_stride() { return 5 * Q + ((5 - 5 * Q) % 8 + 8) % 8; }

// R1 > 1: Q = R1 R2 in two stages; R1 == 1: the R2-point transform in stage A
template <int R1, int R2, class S, int SG, bool EVEN, int TH, int FM>
__global__ void __launch_bounds__(TH) coset_readout_kernel(CosetArgs a)
{
    constexpr int Q = R1 * R2, L = kP * Q, N = 10 * L, FS = frame_stride<Q>();
    constexpr bool kSplit = R1 > 1;
    // with 2 x 11 points the lanes run over the frames first (8-bit samples in
    // stage A, both types in B): a frame's 10 items of B would leave every
    // 8-lane phase two entries on one bank (212 -> 207 us)
    constexpr bool kFrameFastA = R2 == 11 && kSplit && sizeof(S) == 1, kFrameFastB = R2 == 11 && kSplit;
    extern __shared__ __align__(16) unsigned char sm[];
    tc::pdl_start();
    float4* twN = reinterpret_cast<float4*>(sm + a.sm_twN);    // [L / 2] W_N^{r m}: re, re', im, im'
    float4* twL = reinterpret_cast<float4*>(sm + a.sm_twL);    // [Q][5] W_L^{u a}, a = 2 p, 2 p + 1
    float2* twQ = reinterpret_cast<float2*>(sm + a.sm_twQ);    // [R2][R1] cos, sin of 2 pi n2 k1 / Q
    int2* tooth = reinterpret_cast<int2*>(sm + a.sm_tooth);    // [L] tooth of bin (or -1), 1 / reference
    uint64_t* bar = reinterpret_cast<uint64_t*>(sm + a.sm_bar);
    S* raw = reinterpret_cast<S*>(sm + a.sm_raw);
    float4* Y = reinterpret_cast<float4*>(sm + a.sm_Y);
    const S* frames = static_cast<const S*>(a.frames);
    const int T = a.T, F = a.F;
    const int64_t nb = (a.n_frames + F - 1) / F;

    // the copy of batch b: the 16-byte window around its samples (the frames
    // follow one another), but for chunks that would leave the buffer, which
    // go by plain loads
    const uintptr_t buf_lo = reinterpret_cast<uintptr_t>(frames);
    const uintptr_t buf_hi = buf_lo + static_cast<uintptr_t>(a.n_frames) * N * sizeof(S);
    auto issue = [&](int64_t b) {
        const int64_t left = a.n_frames - b * F;
        const uintptr_t p = buf_lo + static_cast<uintptr_t>(b * F) * N * sizeof(S);
        const uintptr_t pe = p + static_cast<uintptr_t>(left < F ? left : F) * N * sizeof(S);
        const uintptr_t p16 = p & ~static_cast<uintptr_t>(15);
        uintptr_t lo = p16, hi = (pe + 15) & ~static_cast<uintptr_t>(15);
        if (lo < buf_lo) {
            lo += 16;
            for (uintptr_t e = p; e < lo; e += sizeof(S)) raw[(e - p16) / sizeof(S)] = *reinterpret_cast<const S*>(e);
        }
        if (hi > buf_hi) {
            hi -= 16;
            for (uintptr_t e = hi; e < pe; e += sizeof(S)) raw[(e - p16) / sizeof(S)] = *reinterpret_cast<const S*>(e);
        }
        tc::fence_proxy_async_smem();   // the batch before was read before this copy is written
        tc::mbar_arrive_expect_tx(bar, static_cast<uint32_t>(hi - lo));
        tc::bulk_g2s(reinterpret_cast<unsigned char*>(raw) + (lo - p16), reinterpret_cast<const void*>(lo),
                     static_cast<uint32_t>(hi - lo), bar);
    };
    int64_t b = blockIdx.x;
    if (threadIdx.x == 0) {
        tc::mbar_init(bar, 1);
        tc::fence_mbar_init();
        if (b < nb) issue(b);
    }
    for (int i = threadIdx.x; i < L / 2; i += TH) {
        const float2 t0 = a.twN[2 * i], t1 = a.twN[2 * i + 1];
        twN[i] = make_float4(t0.x, t1.x, t0.y, t1.y);
    }
    for (int i = threadIdx.x; i < Q * kHalf; i += TH) {
        const int u = i / kHalf, p = i - u * kHalf;
        const float2 t0 = a.twL[u * 2 * p], t1 = a.twL[u * (2 * p + 1)];
        twL[i] = make_float4(t0.x, t1.x, t0.y, t1.y);
    }
    if constexpr (kSplit)
        for (int i = threadIdx.x; i < Q; i += TH) {
            const int e = (i / R1) * (i % R1);
            twQ[i] = make_float2(kRoots<Q>.c[e], kRoots<Q>.s[e]);
        }
    for (int i = threadIdx.x; i < L; i += TH) {
        const int k = a.tooth_of_m[i];
        tooth[i] = make_int2(k, k >= 0 ? __float_as_int(a.inv_ref[k]) : 0);
    }
    const float c1 = a.twM[1].x, s1 = a.twM[1].y, c2 = a.twM[2].x, s2 = a.twM[2].y;
    __syncthreads();

    bool failed = false;
    for (uint32_t phase = 0; b < nb; b += gridDim.x, phase ^= 1u) {
        const int64_t f0 = b * F;
        const int nf = static_cast<int>((a.n_frames - f0) < F ? (a.n_frames - f0) : F);
        // (the barrier also keeps stage A's stores behind the stage C before)
        const bool ok = tc::mbar_wait(bar, phase, 1u << 24);
        if (__syncthreads_or(!ok)) {
            failed = true;
            break;
        }
        const S* xb = raw + ((buf_lo + static_cast<uintptr_t>(f0) * N * sizeof(S)) & 15) / sizeof(S);
        // ---------------- stage A ----------------
        if constexpr (kSplit) {
            constexpr int kItems = kHalf * R2;
            for (int item = threadIdx.x; item < (kFrameFastA ? FM : nf) * kItems; item += TH) {
                const int f = kFrameFastA ? item % FM : item / kItems;
                const int j = kFrameFastA ? item / FM : item % kItems;   // j = p + 5 n2
                if (kFrameFastA && f >= nf) continue;
                const int n2 = j / kHalf;
                C2 z[R1];
#pragma unroll
                for (int n1 = 0; n1 < R1; ++n1)
                    z[n1] = fold_pair<L, S, SG, EVEN>(xb + f * N + 2 * j + kP * R2 * n1, twN[j + kHalf * R2 * n1], c1, s1,
                                                      c2, s2);
                PairDft<R1>::run(z);
                float4* y = Y + f * FS + j + n2 * kHalf * (R1 - 1);   // place (k1 + R1 n2, p)
                y[0] = pack(z[0]);
#pragma unroll
                for (int k1 = 1; k1 < R1; ++k1) {
                    const float2 w = twQ[n2 * R1 + k1];
                    y[kHalf * k1] = pack(crot2(z[k1], dup2(w.x), dup2(w.y)));
                }
            }
        } else {
            for (int item = threadIdx.x; item < nf * kHalf; item += TH) {
                const int f = item / kHalf, p = item - f * kHalf;
                C2 z[Q];
#pragma unroll
                for (int q = 0; q < Q; ++q)
                    z[q] = fold_pair<L, S, SG, EVEN>(xb + f * N + 2 * p + kP * q, twN[p + kHalf * q], c1, s1, c2, s2);
                PairDft<Q>::run(z);
                float4* y = Y + f * FS + p;
                y[0] = pack(z[0]);
#pragma unroll
                for (int u = 1; u < Q; ++u) {
                    const C2 t = unpack(twL[u * kHalf + p]);
                    y[u * kHalf] = pack(cmul2(z[u], t.re, t.im));
                }
            }
        }
        __syncthreads();
        // the samples are read: the next batch's may come
        if (threadIdx.x == 0 && b + gridDim.x < nb) issue(b + gridDim.x);
        // ---------------- stage B ----------------
        if constexpr (kSplit) {
            constexpr int kItems = kHalf * R1;
            for (int item = threadIdx.x; item < (kFrameFastB ? FM : nf) * kItems; item += TH) {
                const int f = kFrameFastB ? item % FM : item / kItems;
                const int j = kFrameFastB ? item / FM : item % kItems;   // j = p + 5 k1
                if (kFrameFastB && f >= nf) continue;
                float4* y = Y + f * FS + j;
                C2 z[R2];
#pragma unroll
                for (int n2 = 0; n2 < R2; ++n2) z[n2] = unpack(y[n2 * R1 * kHalf]);
                PairDft<R2>::run(z);
#pragma unroll
                for (int k2 = 0; k2 < R2; ++k2) {   // u = k1 + R1 k2 (u = 0: times one)
                    const C2 t = unpack(twL[k2 * R1 * kHalf + j]);
                    y[k2 * R1 * kHalf] = pack(cmul2(z[k2], t.re, t.im));
                }
            }
            __syncthreads();
        }
        // ---------------- stage C: Dft<10> over a, its two 5-point halves a pair ----------------
        for (int item = threadIdx.x; item < nf * Q; item += TH) {
            const int f = item / Q, u = item - f * Q;
            const float4* y = Y + f * FS + u * kHalf;
            float zr[kP], zi[kP];
#pragma unroll
            for (int p = 0; p < kHalf; ++p) {
                const float4 v = y[p];
                zr[2 * p] = v.x;
                zr[2 * p + 1] = v.y;
                zi[2 * p] = v.z;
                zi[2 * p + 1] = v.w;
            }
            constexpr RootTable<kP> tab{};
            C2 w[kHalf];
#pragma unroll
            for (int n = 0; n < kHalf; ++n) {
                const float dr = __fsub_rn(zr[n], zr[5 + n]), di = __fsub_rn(zi[n], zi[5 + n]);
                w[n].re.x = __fadd_rn(zr[n], zr[5 + n]);
                w[n].im.x = __fadd_rn(zi[n], zi[5 + n]);
                w[n].re.y = n ? fmaf(dr, tab.c[n], __fmul_rn(di, tab.s[n])) : dr;
                w[n].im.y = n ? fmaf(di, tab.c[n], __fmul_rn(-dr, tab.s[n])) : di;
            }
            PairDft<kHalf>::run(w);
            // straight to global memory: the items of a frame hold runs of
            // consecutive bins, i.e. runs of consecutive (or reversed) teeth
            float* am = a.amps ? a.amps + (f0 + f) * T : nullptr;
            float* yo = a.y ? a.y + (f0 + f) * T : nullptr;
#pragma unroll
            for (int v = 0; v < kP; ++v) {
                const int2 e = tooth[u + Q * v];
                if (e.x >= 0) {
                    const float2 re = w[v / 2].re, im = w[v / 2].im;
                    const float av = cabs_approx((v & 1) ? make_float2(re.y, im.y) : make_float2(re.x, im.x));
                    if (am) am[e.x] = av;
                    if (yo) yo[e.x] = __fmul_rn(av, __int_as_float(e.y));
                }
            }
        }
    }
    if (failed && threadIdx.x == 0) {
        if (a.err) atomicExch(a.err, 3);
        (void)tc::mbar_wait(bar, 0, 1u << 22);   // no copy may land after the block exits
        (void)tc::mbar_wait(bar, 1, 1u << 22);
    }
}

// The instantiated readouts: threads and frames per block, chosen so that the
// stages' items fill the threads and 10 to 20 warps fit an SM.  Measured per
// process call, the readout's share of it changing alone: 1,100 samples, 11
// frames on 64 threads 925 us, 23 on 128 923, 16 on 96 937, 12 on 128 969, 6 on
// 32 1,017; 2,500 samples, 5 on 128 264 us, 10 on 256 266, 7 on 192 266, 4 on
// 128 274, 10 on 128 271, 5 on 64 283; 8-bit, 11 on 128 544 us, 10 on 128 549,
// 11 on 192 562, 6 on 64 598, the 22-point transform in one stage 577 to 644.
struct CosetInst {
    int Q, R1, sb, threads, F;
    void* (*fn)(int sign, bool even);
};
template <int R1, int R2, class S, int TH, int FM>
void* coset_fn(int sign, bool even)
{
    if constexpr (sizeof(S) == 1) {
        if (!even)
            return sign < 0 ? reinterpret_cast<void*>(&coset_readout_kernel<R1, R2, S, -1, false, TH, FM>)
                            : reinterpret_cast<void*>(&coset_readout_kernel<R1, R2, S, 1, false, TH, FM>);
    }
    return sign < 0 ? reinterpret_cast<void*>(&coset_readout_kernel<R1, R2, S, -1, true, TH, FM>)
                    : reinterpret_cast<void*>(&coset_readout_kernel<R1, R2, S, 1, true, TH, FM>);
}
template <int R1, int R2, class S, int TH, int FM>
constexpr CosetInst inst()
{
    return {R1 * R2, R1, static_cast<int>(sizeof(S)), TH, FM, coset_fn<R1, R2, S, TH, FM>};
}
const CosetInst kCoset[] = {
    inst<1, 10, int16_t, 64, 12>(), inst<1, 11, int16_t, 64, 11>(), inst<2, 11, int16_t, 128, 11>(),
    inst<5, 5, int16_t, 128, 5>(),  inst<2, 11, int8_t, 128, 11>(),
};
const CosetInst* find_coset(int Q, int sb)
{
    for (const CosetInst& c : kCoset)
        if (c.Q == Q && c.sb == sb) return &c;
    return nullptr;
}
int align16(int v) { return (v + 15) & ~15; }

}  // namespace

bool coset_instantiated(int Q, int sample_bytes) { return find_coset(Q, sample_bytes) != nullptr; }

// Layout and grid for samples of sb bytes; *grid stays 0 if no block fits.
cudaError_t setup_coset(const cg_plan_s* p, int Q, int sb, CosetArgs& a, int* grid)
{
    const CosetInst* c = find_coset(Q, sb);
    *grid = 0;
    if (!c) return cudaSuccess;
    const int L = kP * Q, N = 10 * L;
    a.T = p->T;
    a.F = c->F;
    int off = 0;
    a.sm_twN = off; off += 8 * L;
    a.sm_twL = off; off += 16 * kHalf * Q;
    a.sm_twQ = off; off = align16(off + (c->R1 > 1 ? 8 * Q : 0));
    a.sm_tooth = off; off = align16(off + 8 * L);
    a.sm_bar = off; off += 16;
    a.sm_raw = off; off += align16(sb * N * c->F) + 16;
    const int fs = 5 * Q + ((5 - 5 * Q) % 8 + 8) % 8;
    a.sm_Y = off; off += 16 * fs * c->F;
    a.sm_total = off;
    a.twL = p->d.tw_L;
    a.twN = p->d.tw_n1;
    a.twM = p->d.tw_M5;
    a.tooth_of_m = p->d.tooth_of_m;
    a.inv_ref = p->d.inv_ref;
    const int sign = (p->r0 & 1) ? -1 : 1;
    int most = 1 << 30;
    for (bool even : {true, false}) {
        void* fn = c->fn(sign, even);
        cudaError_t e = raise_smem_limit(fn, a.sm_total);
        if (e != cudaSuccess) return e;
        int occ = 0;
        if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, fn, c->threads, a.sm_total)) != cudaSuccess) return e;
        most = std::min(most, occ);
    }
    *grid = p->num_sms * most;
    return cudaSuccess;
}

static cudaError_t launch_coset(const cg_plan_s* p, const void* frames, int sb, int64_t n, float* amps, float* y,
                                cudaStream_t s)
{
    const CosetInst* c = find_coset(p->Q, sb);
    if (!c) return cudaErrorInvalidValue;
    CosetArgs a = sb == 1 ? p->fa8 : p->fa;
    // every block takes the same number of batches: of so many frames that the
    // last round is as full as the others, and few frames lie on all SMs
    const int gmax = sb == 1 ? p->grid_fast8 : p->grid_fast;
    const int64_t rounds = (n + static_cast<int64_t>(gmax) * a.F - 1) / (static_cast<int64_t>(gmax) * a.F);
    a.F = static_cast<int>((n + gmax * rounds - 1) / (gmax * rounds));
    a.frames = frames;
    a.n_frames = n;
    a.amps = amps;
    a.y = y;
    a.err = p->d.err;
    const int64_t nb = (n + a.F - 1) / a.F;
    const int grid = static_cast<int>(nb < gmax ? nb : gmax);
    const bool even = !(reinterpret_cast<uintptr_t>(frames) & 1);
    void* args[] = {&a};
    return cudaLaunchKernel(c->fn((p->r0 & 1) ? -1 : 1, even), dim3(grid), dim3(c->threads), args, a.sm_total, s);
}

cudaError_t launch_fast_readout(const cg_plan_s* p, const int16_t* frames, int64_t n, float* amps, float* y,
                                cudaStream_t s)
{
    return launch_coset(p, frames, 2, n, amps, y, s);
}

cudaError_t launch_fast_readout_i8(const cg_plan_s* p, const int8_t* frames, int64_t n, float* amps, float* y,
                                   cudaStream_t s)
{
    return launch_coset(p, frames, 1, n, amps, y, s);
}

}  // namespace cg
