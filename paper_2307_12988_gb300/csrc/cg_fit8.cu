// cg_fit8.cu -- the standalone Levenberg-Marquardt fit at eight lanes per
// frame (cg_fit, and the fit of CG_PATH_SPLIT) of more spectra than the groups
// of fit_kernel hold at once, two or four frames per lane group.
//
// Paper ("Data Capture and Processing", fit paragraphs): each normalised
// spectrum is fit by Levenberg-Marquardt, at most 20 iterations, tolerance
// 1e-6.  Arithmetic, sums and decisions are those of fit_group<8>
// (cg_fit.cuh): lane l of a frame's eight adds up teeth l, l + 8, ... in
// order, the eight partial sums are added over lane distances 4, 2, 1.  What
// differs is how the work lies on the warp:
//  * a group of eight lanes evaluates two (or two pairs of) frames at once, one
//    in each half of packed FP32x2 operations;
//  * the exchanges over distances 4 and 2 also sort the 14 sums by frame: they
//    end in the four (two) lanes that own it, so one pass of the 4 x 4 solve
//    and of the decisions serves every frame of the group -- eight (sixteen)
//    per warp, where every lane of a group repeated one frame's;
//  * each owner pulls its next frame when its own is done; the row arrives
//    meanwhile by one bulk copy into the owner's other slot, so no frame waits
//    for another's iterations;
//  * the moment guess runs before, one lane per frame (init_kernel), and
//    leaves its starting point (normalised abscissa) in params.
//
// What bounds it: instruction issue (two frames a group: 65 % active; about 970
// warp instructions per evaluation of eight frames of 99 teeth, 390 of them in
// the teeth's loop, where fit_group spent 1,340 on two times four; four a
// group: about 1,350 for sixteen).  10^5 spectra of 99 teeth: 159 us in
// fit_kernel, which also held every block for its slowest frame; 88 us with
// two frames a group, 84 with four, and 10 to 17 for the guess.
#include <algorithm>
#include <cstdint>
#include <cuda_runtime.h>

#include "cg_fit.cuh"
#include "cg_internal.h"
#include "cg_tc.cuh"

namespace cg {

namespace {

constexpr int kWarps8 = 4;       // warps per block

__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 neg2(float2 a) { return make_float2(-a.x, -a.y); }

struct Fit8Args {
    int64_t n;
    int T, RS, task;                // teeth, slot stride (floats), frames per warp task
    const float* y;                 // [n][T] or null (then amps * inv_ref)
    const float* amps;
    const float* inv_ref;
    const float* u;
    const float* p0;                // [n][4]: abscissa units, or (guessed) on the normalised abscissa
    int guessed;
    unsigned long long* counter;    // see next_task
    float x_mid, x_scale;
    int max_iter;
    float tol, lambda0;
    float *params, *rss;
    int16_t *iters, *status;
    int* err;
};

// the 14 sums of accum_point for one tooth of two frames
__device__ __forceinline__ void accum_pair(float u, float2 y, float2 c, float2 g2, float2 nA, float2 nB, float2 (&s)[14])
{
    const float2 d = add2(make_float2(u, u), neg2(c));
    const float2 D = fma2(d, d, g2);
    const float2 q = make_float2(rcp_fast(D.x), rcp_fast(D.y));
    const float2 L = mul2(g2, q);
    const float2 r = fma2(nA, L, add2(y, nB));
    const float2 t = mul2(L, q);
    const float2 jc = mul2(t, d);
    const float2 jg = mul2(jc, d);
    s[0] = fma2(L, L, s[0]);
    s[1] = fma2(L, jc, s[1]);
    s[2] = fma2(L, jg, s[2]);
    s[3] = add2(s[3], L);
    s[4] = fma2(jc, jc, s[4]);
    s[5] = fma2(jc, jg, s[5]);
    s[6] = add2(s[6], jc);
    s[7] = fma2(jg, jg, s[7]);
    s[8] = add2(s[8], jg);
    s[9] = fma2(L, r, s[9]);
    s[10] = fma2(jc, r, s[10]);
    s[11] = fma2(jg, r, s[11]);
    s[12] = add2(s[12], r);
    s[13] = fma2(r, r, s[13]);
}

// sums over the eight lanes, distances 4, 2, 1.  Two frames: the lower four
// lanes get the first frame's 14 sums, the upper four the second's
__device__ __forceinline__ void reduce_frames(const float2 (&s2)[1][14], LmSums& S)
{
    const float2 (&s)[14] = s2[0];
    const int lane = threadIdx.x & 31;
    const bool hi = (lane & 4) != 0;
    float a[14];
#pragma unroll
    for (int i = 0; i < 14; ++i) {
        const float send = hi ? s[i].x : s[i].y, keep = hi ? s[i].y : s[i].x;
        a[i] = keep + __shfl_xor_sync(kFull, send, 4);
    }
    // distance 2: each keeps seven; distance 1: four or three of those
    const bool b2 = (lane & 2) != 0;
    float b[8];
#pragma unroll
    for (int i = 0; i < 7; ++i) {
        const float send = b2 ? a[i] : a[i + 7], keep = b2 ? a[i + 7] : a[i];
        b[i] = keep + __shfl_xor_sync(kFull, send, 2);
    }
    b[7] = 0.f;
    const bool b1 = (lane & 1) != 0;
    float c[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const float send = b1 ? b[i] : b[i + 4], keep = b1 ? b[i + 4] : b[i];
        c[i] = keep + __shfl_xor_sync(kFull, send, 1);
    }
    const int base = lane & ~3;
#pragma unroll
    for (int i = 0; i < 14; ++i) {
        const int in7 = i % 7, owner = (i / 7) * 2 + in7 / 4;
        S.v[i] = __shfl_sync(kFull, c[in7 % 4], base + owner);
    }
}

// Four frames (the first two in s[0], the others in s[1]): two lanes each
__device__ __forceinline__ void reduce_frames(const float2 (&s)[2][14], LmSums& S)
{
    const int lane = threadIdx.x & 31;
    const bool b4 = (lane & 4) != 0, b2 = (lane & 2) != 0;
#pragma unroll
    for (int i = 0; i < 14; ++i) {
        const float2 send = b4 ? s[0][i] : s[1][i], keep = b4 ? s[1][i] : s[0][i];
        const float2 got = make_float2(__shfl_xor_sync(kFull, send.x, 4), __shfl_xor_sync(kFull, send.y, 4));
        const float2 a = make_float2(keep.x + got.x, keep.y + got.y);
        const float b = (b2 ? a.y : a.x) + __shfl_xor_sync(kFull, b2 ? a.x : a.y, 2);
        S.v[i] = b + __shfl_xor_sync(kFull, b, 1);
    }
}

// NF: frames of a lane group (2 or 4); 8 / NF lanes own a frame
template <bool SCALE, int NF>
__global__ void __launch_bounds__(32 * kWarps8, NF == 2 ? 4 : 3) fit8_kernel(Fit8Args a)
{
    constexpr int LP = 8 / NF;               // lanes that own a frame
    constexpr int kInFlight = 32 / LP;       // frames of a warp
    constexpr int kSlots8 = 2 * kInFlight;   // its row slots
    extern __shared__ __align__(16) float f8sm[];
    const int T = a.T;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int gl = lane & 7, own = lane & (LP - 1), leader = lane & ~(LP - 1), half = lane / LP;   // half: the frame
    // its slot of either parity: those that the four groups read at a time lie
    // a quarter of the banks apart (row stride 24 mod 32 for two slots, 8 or 24
    // for one)
    const int place = NF == 2 ? half : (half >> 2) + 4 * (half & 3);
    float* slots = f8sm + warp * kSlots8 * a.RS;
    uint64_t* bars = reinterpret_cast<uint64_t*>(f8sm + kWarps8 * kSlots8 * a.RS) + warp * kSlots8;
    float* us = reinterpret_cast<float*>(reinterpret_cast<uint64_t*>(f8sm + kWarps8 * kSlots8 * a.RS) + kWarps8 * kSlots8);
    float* iref = us + T;
    for (int i = threadIdx.x; i < T; i += blockDim.x) {
        us[i] = a.u[i];
        iref[i] = SCALE ? a.inv_ref[i] : 1.0f;
    }
    // (a half without a frame evaluates whatever its slot holds: finite values)
    for (int i = threadIdx.x; i < kWarps8 * kSlots8 * a.RS; i += blockDim.x) f8sm[i] = 0.f;
    if (lane < kSlots8) tc::mbar_init(&bars[lane], 1);
    tc::fence_mbar_init();
    tc::fence_proxy_async_smem();
    __syncthreads();
    tc::pdl_wait();

    const float* src_base = SCALE ? a.amps : a.y;
    const uintptr_t buf_lo = reinterpret_cast<uintptr_t>(src_base);
    const uintptr_t buf_hi = buf_lo + static_cast<uintptr_t>(a.n) * T * sizeof(float);
    const int64_t n = a.n;
    // the warp's tasks, the current one [next, end)
    bool first = true;
    int64_t next = 0, end = 0;
    int64_t f = -1, fn = -1;     // frame being fit; next frame (its copy in flight)
    float pn[4] = {0.f, 1.f, 0.f, 0.f};
    int cs = 0, oc = 0, on = 0;
    uint32_t ph = 0;
    float p[4] = {0.f, 1.f, 0.f, 0.f};
    float lambda = a.lambda0, chi2 = 0.f;
    Normal Nm;
#pragma unroll
    for (int i = 0; i < 10; ++i) Nm.H[i] = 0.f;
#pragma unroll
    for (int i = 0; i < 4; ++i) Nm.b[i] = 0.f;
    int it = 0, st = kMaxIter, flag = 0;
    bool fresh = false, failed = false;

    while (true) {
        // ---- a half without a frame starts its next one ----
        if (f < 0 && fn >= 0) {
            const int nx = cs ^ 1;
            const int sl = place + kInFlight * nx;
            if (!tc::mbar_wait(&bars[sl], (ph >> nx) & 1u, 1u << 22)) failed = true;
            ph ^= 1u << nx;
            cs = nx;
            f = fn;
            oc = on;
            fn = -1;
            fresh = true;
            flag = 0;
            if (a.guessed) {
#pragma unroll
                for (int i = 0; i < 4; ++i) p[i] = pn[i];
                flag = pn[2] == 0.f ? kInitFlat : 0;   // (only a flat spectrum's guess has no amplitude)
            } else {
                p[0] = (pn[0] - a.x_mid) / a.x_scale;
                p[1] = pn[1] / a.x_scale;
                p[2] = pn[2];
                p[3] = pn[3];
            }
            lambda = a.lambda0;
            it = 0;
            st = kMaxIter;
        }
        if (__any_sync(kFull, failed)) break;
        // ---- halves without a next frame claim one; its row goes to the free slot ----
        unsigned need = __ballot_sync(kFull, own == 0 && fn < 0);
        while (need != 0 && next < n) {
            if (next >= end) {
                next = next_task(a.counter, first, warp * gridDim.x + blockIdx.x, kWarps8 * gridDim.x, a.task, end, n);
                if (next >= n) {
                    next = end = n;
                    break;
                }
                end = next + a.task < n ? next + a.task : n;
            }
            const int cnt = __popc(need);
            const int64_t avail = end - next;
            const int take = static_cast<int>(avail < cnt ? avail : cnt);
            const int rank = __popc(need & ((1u << leader) - 1u));
            if (((need >> leader) & 1u) && rank < take) {
                fn = next + rank;
                const float* q = a.p0 + fn * 4;
#pragma unroll
                for (int i = 0; i < 4; ++i) pn[i] = q[i];
                const float* src = src_base + fn * T;
                const uintptr_t ad = reinterpret_cast<uintptr_t>(src);
                const uintptr_t a16 = ad & ~static_cast<uintptr_t>(15);
                const uintptr_t e16 = (ad + 4u * T + 15u) & ~static_cast<uintptr_t>(15);
                on = static_cast<int>((ad - a16) >> 2);
                const int sl = place + kInFlight * (cs ^ 1);
                float* dst = slots + sl * a.RS;
                if (own == 0) {
                    if (a16 >= buf_lo && e16 <= buf_hi) {
                        tc::fence_proxy_async_smem();   // the slot's last reads precede this write
                        tc::mbar_arrive_expect_tx(&bars[sl], static_cast<uint32_t>(e16 - a16));
                        tc::bulk_g2s(dst, reinterpret_cast<const void*>(a16), static_cast<uint32_t>(e16 - a16), &bars[sl]);
                    } else {
                        // the first or last row of an unaligned buffer: its
                        // window would leave the buffer
                        for (int k = 0; k < T; ++k) dst[on + k] = src[k];
                        tc::mbar_arrive(&bars[sl]);
                    }
                }
            }
            next += take;
            need = __ballot_sync(kFull, own == 0 && fn < 0);
        }
        if (!__any_sync(kFull, f >= 0 || fn >= 0)) break;

        // ---- trial point of this half's frame ----
        float pt[4] = {p[0], p[1], p[2], p[3]};
        bool done = false;
        if (f >= 0 && !fresh) {
            float delta[4] = {0.f, 0.f, 0.f, 0.f};
            if (lm_solve4(Nm, lambda, delta)) {
#pragma unroll
                for (int i = 0; i < 4; ++i) pt[i] = __fadd_rn(p[i], delta[i]);
            } else {
                st = kSingular;
                done = true;
            }
        }
        // ---- sums of both frames of the group at their trial points ----
        float2 s[NF / 2][14];
        {
            // the group's frames: (first, second), (third, fourth)
            const int base = lane & ~7;
            auto pairs = [&](float v, float2 (&o)[NF / 2]) {
                if constexpr (NF == 2) {
                    const float w = __shfl_xor_sync(kFull, v, 4);
                    o[0] = (lane & 4) ? make_float2(w, v) : make_float2(v, w);
                } else {
#pragma unroll
                    for (int h = 0; h < NF / 2; ++h)
                        o[h] = make_float2(__shfl_sync(kFull, v, base + 2 * LP * h), __shfl_sync(kFull, v, base + 2 * LP * h + LP));
                }
            };
            float2 c[NF / 2], g2[NF / 2], nA[NF / 2], nB[NF / 2];
            pairs(pt[0], c);
            pairs(pt[1] * pt[1], g2);
            pairs(-pt[2], nA);
            pairs(-pt[3], nB);
            const int mine = (place + kInFlight * cs) * a.RS + oc;
            const float* row[NF];
#pragma unroll
            for (int q = 0; q < NF; ++q) row[q] = slots + __shfl_sync(kFull, mine, base + LP * q);
#pragma unroll
            for (int h = 0; h < NF / 2; ++h)
#pragma unroll
                for (int i = 0; i < 14; ++i) s[h][i] = make_float2(0.f, 0.f);
#pragma unroll 2
            for (int k = gl; k < T; k += 8) {
                const float uk = us[k], ik = SCALE ? iref[k] : 1.f;
#pragma unroll
                for (int h = 0; h < NF / 2; ++h) {
                    float2 y = make_float2(row[2 * h][k], row[2 * h + 1][k]);
                    if (SCALE) y = make_float2(__fmul_rn(y.x, ik), __fmul_rn(y.y, ik));
                    accum_pair(uk, y, c[h], g2[h], nA[h], nB[h], s[h]);
                }
            }
        }
        LmSums S;
        reduce_frames(s, S);
        // ---- decisions (as fit_group) ----
        if (f >= 0 && !done) {
            const float chi2t = S.v[13];
            if (fresh) {
                chi2 = chi2t;
                make_normal(S, pt[1], pt[2], T, Nm);
                if (!(chi2t < INFINITY)) {
                    st = kNonfinite;
                    done = true;
                }
                if (a.max_iter <= 0) done = true;
            } else {
                ++it;
                if (!(chi2t < INFINITY)) {
                    lambda *= 10.0f;
                } else if (chi2_settled(chi2t, chi2, a.tol, p[2], p[3])) {
                    if (chi2t <= chi2) {
#pragma unroll
                        for (int i = 0; i < 4; ++i) p[i] = pt[i];
                        chi2 = chi2t;
                    }
                    st = kConverged;
                    done = true;
                } else if (chi2t < chi2) {
#pragma unroll
                    for (int i = 0; i < 4; ++i) p[i] = pt[i];
                    chi2 = chi2t;
                    make_normal(S, pt[1], pt[2], T, Nm);
                    lambda *= 0.1f;
                } else {
                    lambda *= 10.0f;
                }
                if (!done && it >= a.max_iter) done = true;
            }
        }
        fresh = false;
        if (f >= 0 && done) {
            if (own == 0) {
                float* po = a.params + f * 4;
                po[0] = fmaf(a.x_scale, p[0], a.x_mid);
                po[1] = a.x_scale * fabsf(p[1]);
                po[2] = p[2];
                po[3] = p[3];
                if (a.rss) a.rss[f] = chi2;
                if (a.iters) a.iters[f] = static_cast<int16_t>(it);
                if (a.status) a.status[f] = static_cast<int16_t>(st | flag);
            }
            f = -1;
        }
    }
    // no copy may land after the block exits (a failed wait only)
    if (fn >= 0) {
        const int nx = cs ^ 1;
        tc::mbar_wait(&bars[place + kInFlight * nx], (ph >> nx) & 1u, 1u << 22);
    }
    if (failed && lane == 0 && a.err) atomicExch(a.err, 4);
}

// floats of the largest 16-byte window around a row, as a stride: an odd
// multiple of 4 (two frames a group) or of 8 (four)
int row_window(int T, int frames)
{
    const int step = 2 * frames, w = (4 * T + 12 + 15) / 16 * 4;
    return (w + step - 1) / step * step + ((w + step - 1) / step % 2 ? 0 : step);
}
int fit8_slots(int frames) { return 2 * 4 * frames; }   // per warp
int fit8_smem(int T, int frames) { return kWarps8 * fit8_slots(frames) * (4 * row_window(T, frames) + 8) + 8 * T; }
void* fit8_fn(bool scale, int frames)
{
    if (frames == 4)
        return scale ? reinterpret_cast<void*>(&fit8_kernel<true, 4>) : reinterpret_cast<void*>(&fit8_kernel<false, 4>);
    return scale ? reinterpret_cast<void*>(&fit8_kernel<true, 2>) : reinterpret_cast<void*>(&fit8_kernel<false, 2>);
}

}  // namespace

cudaError_t setup_fit8(cg_plan_s* p)
{
    p->fit8_ok = false;
    if (p->G != 8 || !p->fit_ok) return cudaSuccess;
    int most = 0;
    cudaError_t e = cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin, p->device);
    if (e != cudaSuccess) return e;
    // blocks per SM with n frames in a lane group (0: they don't fit)
    auto blocks = [&](int frames, int* occ) -> cudaError_t {
        const int bytes = fit8_smem(p->T, frames);
        *occ = 0;
        if (bytes > most) return cudaSuccess;
        int o[2] = {};
        for (int i = 0; i < 2; ++i) {
            void* fn = fit8_fn(i, frames);
            cudaError_t r = raise_smem_limit(fn, bytes);
            if (r == cudaSuccess) r = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o[i], fn, 32 * kWarps8, bytes);
            if (r != cudaSuccess) return r;
        }
        *occ = std::min(o[0], o[1]);
        return cudaSuccess;
    };
    int occ = 0;
    if ((e = blocks(2, &occ)) != cudaSuccess) return e;
    if (occ < 1) return cudaSuccess;
    p->grid_fit8 = p->num_sms * occ;
    // four frames a group where three blocks' rows fit an SM (fewer warps took
    // longer than two frames a group)
    if ((e = blocks(4, &occ)) != cudaSuccess) return e;
    p->grid_fit8_four = occ >= 3 ? p->num_sms * occ : 0;
    if ((e = raise_smem_limit(init_ptr(p->init_npad, p->n_outer, true), p->init_smem)) != cudaSuccess) return e;
    p->fit8_ok = true;
    return cudaSuccess;
}

cudaError_t launch_fit8(const cg_plan_s* p, const float* y, const float* amps, int64_t n, const float* p0,
                        float* params, float* rss, int16_t* iters, int16_t* status, unsigned long long* counter,
                        cudaStream_t s)
{
    const FitArgs fa = make_fit_args(p);
    if (!p0) {
        const cudaError_t e = launch_init(p, y, amps, n, params, nullptr, s, nullptr, nullptr, true);
        if (e != cudaSuccess) return e;
    }
    // Four frames a group do a third less work per frame but take a third longer
    // per step of all of them, so they pay where two a group would need a good
    // part of a second round of frames (99 teeth, two / four: 20,000 spectra 36 / 42 us, 50,000
    // 70 / 54, 10^5 104 / 99, 400,000 345 / 292; 21 teeth: 20,000 24 / 26,
    // 50,000 48 / 31, 400,000 217 / 171)
    const bool four = p->grid_fit8_four > 0 && 4 * n > 5 * static_cast<int64_t>(p->grid_fit8) * kWarps8 * fit8_slots(2) / 2;
    const int frames = four ? 4 : 2, blocks = four ? p->grid_fit8_four : p->grid_fit8;
    Fit8Args a{};
    a.n = n;
    a.T = p->T;
    a.RS = row_window(p->T, frames);
    // frames per task as in launch_fit3: two per frame in flight, fewer where
    // the schedulers would otherwise have none
    const int64_t schedulers = 4 * static_cast<int64_t>(p->num_sms);
    a.task = static_cast<int>(std::min<int64_t>(fit8_slots(frames), (n + schedulers - 1) / schedulers));
    a.y = y;
    a.amps = amps;
    a.inv_ref = fa.inv_ref;
    a.u = fa.u;
    a.p0 = p0 ? p0 : params;
    a.guessed = p0 ? 0 : 1;
    a.counter = counter;
    a.x_mid = fa.x_mid;
    a.x_scale = fa.x_scale;
    a.max_iter = fa.max_iter;
    a.tol = fa.tol;
    a.lambda0 = fa.lambda0;
    a.params = params;
    a.rss = rss;
    a.iters = iters;
    a.status = status;
    a.err = p->d.err;
    const int64_t tasks = (n + a.task - 1) / a.task;
    const int grid = static_cast<int>(tasks < blocks ? tasks : blocks);
    if (counter && tasks > static_cast<int64_t>(grid) * kWarps8) {
        const cudaError_t e = cudaMemsetAsync(a.counter, 0, sizeof(unsigned long long), s);
        if (e != cudaSuccess) return e;
    }
    void* args[] = {&a};
    return launch_dependent(fit8_fn(!y, frames), dim3(grid), dim3(32 * kWarps8), args, fit8_smem(p->T, frames), s);
}

}  // namespace cg
