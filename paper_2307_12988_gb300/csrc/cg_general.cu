// cg_general.cu -- tooth readout by the general transform: any frame length
// that is a product of 2, 3, 5, 7, 11 and 13 and any tooth bins (the comb
// geometries and power-of-two lengths have kernels of their own).
//
// Paper ("Data Capture and Processing"): each row of N samples is Fourier
// transformed and the tooth bins are read and divided by the reference.
//
// The L complex values of a frame (real-FFT packing z_n = x_2n + i x_2n+1,
// or the coset fold) are transformed in place in shared memory by the plan's
// radices, decimation in time: stage s of radix R combines points S apart,
// S = L / (product of the radices up to s), after multiplying them by
// W^(r k), and writes the results where it read them.  The result is in
// digit-reversed order, which only the table of the teeth's positions knows.
// Two consecutive radices with a product of at most 16 are taken in one pass
// with both butterflies in registers.  The first pass reads the samples as
// they were staged, and the next batch's samples arrive (cp.async) while the
// other passes run.
//
// What bounds it: instruction issue (about 2,300 warp instructions for a
// 2,640-sample frame), so the passes divide by multiplication, twiddles lie
// in the order the threads read them, and the frames per block are chosen to
// leave few threads idle in the passes.  readout_kernel, which it replaces
// for readouts, kept two buffers and staged synchronously.
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <vector>
#include <cuda_runtime.h>

#include "cg_fft.cuh"
#include "cg_internal.h"
#include "cg_stage.cuh"
#include "cg_tc.cuh"

namespace cg {

namespace {

constexpr int kGenThreads = 128;

// place of point p: with a power-of-two last radix one pad per 16 points
// keeps its butterflies (R points apart) off each other's banks
template <bool PAD>
__device__ __forceinline__ int gp(int p) { return PAD ? p + (p >> 4) : p; }

// v / d with magic = floor(2^32 / d) + 1 (0 for d = 1), exact for v d < 2^32
__device__ __forceinline__ int div_by(int v, uint32_t magic)
{
    return magic ? static_cast<int>(__umulhi(static_cast<uint32_t>(v), magic)) : v;
}

// radices RA then RB (RB = 1: one stage) over nf frames.  kFirst: no twiddles
// on RA, and in RAW form the points come from the samples (the low and high
// half of a 32-bit word where the frames are 4-byte aligned).
template <int RA, int RB, bool PAD, bool RAW>
__device__ __forceinline__ void gen_pass(const GenPass& q, int nf, float2* Z, int zstride, const int16_t* raw, int N,
                                         bool words, const float2* tw)
{
    const int total = nf * q.per;
    for (int item = threadIdx.x; item < total; item += kGenThreads) {
        const int f = div_by(item, q.magic_per);
        const int b = item - f * q.per;
        const int blk = div_by(b, q.magic_s);
        const int j = b - blk * q.s;
        const int base = blk * (q.s * RA * RB) + j;
        float2* Zf = Z + f * zstride;
        float2 a[RB][RA];
#pragma unroll
        for (int rb = 0; rb < RB; ++rb)
#pragma unroll
            for (int ra = 0; ra < RA; ++ra) {
                const int p = base + (ra * RB + rb) * q.s;
                if constexpr (RAW) {
                    const int16_t* xs = raw + f * N + 2 * p;
                    if (words) {
                        const uint32_t w = *reinterpret_cast<const uint32_t*>(xs);
                        a[rb][ra] = make_float2(static_cast<float>(static_cast<short>(w & 0xffffu)),
                                                static_cast<float>(static_cast<short>(w >> 16)));
                    } else {
                        a[rb][ra] = make_float2(static_cast<float>(xs[0]), static_cast<float>(xs[1]));
                    }
                } else {
                    a[rb][ra] = Zf[gp<PAD>(p)];
                }
            }
        if (q.ns > 1) {
            const float2* t = tw + q.off_a + blk;
#pragma unroll
            for (int ra = 1; ra < RA; ++ra) {
                const float2 w = t[(ra - 1) * q.ns];
#pragma unroll
                for (int rb = 0; rb < RB; ++rb) a[rb][ra] = cmul(a[rb][ra], w);
            }
        }
#pragma unroll
        for (int rb = 0; rb < RB; ++rb) Dft<RA>::run(a[rb]);
        if constexpr (RB == 1) {
#pragma unroll
            for (int ra = 0; ra < RA; ++ra) Zf[gp<PAD>(base + ra * q.s)] = a[0][ra];
        } else {
            const float2* t = tw + q.off_b + blk * RA;
#pragma unroll
            for (int ka = 0; ka < RA; ++ka) {
                float2 v[RB];
                v[0] = a[0][ka];
#pragma unroll
                for (int rb = 1; rb < RB; ++rb) v[rb] = cmul(a[rb][ka], t[(rb - 1) * (q.ns * RA) + ka]);
                Dft<RB>::run(v);
#pragma unroll
                for (int rb = 0; rb < RB; ++rb) Zf[gp<PAD>(base + (ka * RB + rb) * q.s)] = v[rb];
            }
        }
    }
}

template <bool PAD, bool RAW>
__device__ __forceinline__ void gen_dispatch(const GenPass& q, int nf, float2* Z, int zstride, const int16_t* raw,
                                             int N, bool words, const float2* tw)
{
#define CG_PASS(A, B)                                                    \
    case 16 * A + B:                                                     \
        gen_pass<A, B, PAD, RAW>(q, nf, Z, zstride, raw, N, words, tw);  \
        break;
    switch (16 * q.ra + q.rb) {
        CG_PASS(2, 1)
        CG_PASS(3, 1)
        CG_PASS(4, 1)
        CG_PASS(5, 1)
        CG_PASS(7, 1)
        CG_PASS(8, 1)
        CG_PASS(11, 1)
        CG_PASS(13, 1)
        CG_PASS(8, 2)
        CG_PASS(4, 2)
        CG_PASS(4, 3)
        CG_PASS(2, 3)
        CG_PASS(2, 5)
        CG_PASS(2, 7)
        CG_PASS(5, 3)
        CG_PASS(3, 3)
    default: break;
    }
#undef CG_PASS
}

template <bool PAD>
__global__ void __launch_bounds__(kGenThreads, 6) general_readout_kernel(const __grid_constant__ GenArgs a)
{
    extern __shared__ __align__(16) unsigned char gsm[];
    tc::pdl_start();
    float2* tw = reinterpret_cast<float2*>(gsm);
    float2* twn1 = reinterpret_cast<float2*>(gsm + a.sm_n1);   // coset: [L] W_N^(r n1), then [M] W_M^(r n2)
    float2* twb = reinterpret_cast<float2*>(gsm + a.sm_b);     // full: [T] W_N^(b_k)
    int2* pos = reinterpret_cast<int2*>(gsm + a.sm_pos);       // [T] places of Z_b and Z_(L - b)
    float* iref = reinterpret_cast<float*>(gsm + a.sm_iref);
    int16_t* raw = reinterpret_cast<int16_t*>(gsm + a.sm_raw);
    float2* Z = reinterpret_cast<float2*>(gsm + a.sm_z);
    const int T = a.T, N = a.N, L = a.L, F = a.F, M = a.M;
    const bool coset = a.kind == CG_FFT_COSET;
    const int64_t nb = (a.n_frames + F - 1) / F;
    auto frames_of = [&](int64_t b) { return static_cast<int>((a.n_frames - b * F) < F ? (a.n_frames - b * F) : F); };
    int64_t b = blockIdx.x;
    int off = 0;
    if (b < nb) off = stage_async(a.frames, b * F * static_cast<int64_t>(N), static_cast<int64_t>(frames_of(b)) * N, raw);
    for (int i = threadIdx.x; i < L; i += kGenThreads) tw[i] = a.tw[i];
    if (coset) {
        for (int i = threadIdx.x; i < L; i += kGenThreads) twn1[i] = a.tw_n1[i];
        for (int i = threadIdx.x; i < M; i += kGenThreads) twn1[L + i] = a.tw_M[i];
    } else {
        for (int i = threadIdx.x; i < T; i += kGenThreads) twb[i] = a.tw_b[i];
    }
    for (int i = threadIdx.x; i < T; i += kGenThreads) {
        pos[i] = a.pos[i];
        iref[i] = a.inv_ref[i];
    }
    for (; b < nb; b += gridDim.x) {
        const int64_t f0 = b * F;
        const int nf = frames_of(b);
        cp_async_wait_all();
        __syncthreads();
        const int16_t* x = raw + off;
        int first = 0;
        if (coset) {
            for (int item = threadIdx.x; item < nf * L; item += kGenThreads) {
                const int f = div_by(item, a.magic_l);
                const int n1 = item - f * L;
                const int16_t* xs = x + f * N + n1;
                float2 acc = make_float2(0.f, 0.f);
                for (int n2 = 0; n2 < M; ++n2) {
                    const float v = static_cast<float>(xs[n2 * L]);
                    const float2 w = twn1[L + n2];
                    acc.x = fmaf(v, w.x, acc.x);
                    acc.y = fmaf(v, w.y, acc.y);
                }
                Z[f * a.zstride + gp<PAD>(n1)] = cmul(acc, twn1[n1]);
            }
        } else {
            gen_dispatch<PAD, true>(a.pass[0], nf, Z, a.zstride, x, N, (off & 1) == 0, tw);
            first = 1;
        }
        __syncthreads();
        // the samples are used up: the next batch's arrive meanwhile
        const int64_t bn = b + gridDim.x;
        if (bn < nb)
            off = stage_async(a.frames, bn * F * static_cast<int64_t>(N), static_cast<int64_t>(frames_of(bn)) * N, raw);
        for (int s = first; s < a.npass; ++s) {
            gen_dispatch<PAD, false>(a.pass[s], nf, Z, a.zstride, nullptr, N, false, tw);
            __syncthreads();
        }
        // teeth
        for (int item = threadIdx.x; item < nf * T; item += kGenThreads) {
            const int f = div_by(item, a.magic_t);
            const int k = item - f * T;
            const float2* Zf = Z + f * a.zstride;
            const int2 p = pos[k];
            float2 X;
            if (coset) {
                X = Zf[p.x];
            } else {
                const float2 Zb = Zf[p.x];
                const float2 Zr = Zf[p.y];
                // even part E = (Zb + conj Zr)/2, odd part O = (Zb - conj Zr)/(2i)
                const float2 E = make_float2(0.5f * (Zb.x + Zr.x), 0.5f * (Zb.y - Zr.y));
                const float2 Dd = make_float2(0.5f * (Zb.x - Zr.x), 0.5f * (Zb.y + Zr.y));
                X = cadd(E, cmul(twb[k], make_float2(Dd.y, -Dd.x)));
            }
            const float amp = sqrtf(fmaf(X.x, X.x, X.y * X.y));
            const int64_t o = (f0 + f) * T + k;
            if (a.amps) a.amps[o] = amp;
            if (a.y) a.y[o] = __fmul_rn(amp, iref[k]);
        }
    }
    cp_async_wait_all();
}

void* gen_ptr(bool pad)
{
    return pad ? reinterpret_cast<void*>(&general_readout_kernel<true>)
               : reinterpret_cast<void*>(&general_readout_kernel<false>);
}

uint32_t magic_of(int d) { return d > 1 ? static_cast<uint32_t>((uint64_t(1) << 32) / static_cast<uint32_t>(d)) + 1u : 0u; }

// pairs of radices that are taken in one pass
bool fusable(int ra, int rb)
{
    static const int kPairs[][2] = {{8, 2}, {4, 2}, {4, 3}, {2, 3}, {2, 5}, {2, 7}, {5, 3}, {3, 3}};
    for (const auto& q : kPairs)
        if (q[0] == ra && q[1] == rb) return true;
    return false;
}

int align16(int v) { return (v + 15) & ~15; }

}  // namespace

// Passes, tables and layout of the general readout for the plan's transform
// (p->ra holds its radices and tables); zidx as in ReadoutArgs.
cudaError_t setup_general(cg_plan_s* p, const std::vector<int>& zidx)
{
    GenArgs& g = p->ga_gen;
    const ReadoutArgs& r = p->ra;
    const int L = r.L, T = r.T, N = r.N;
    g.N = N;
    g.T = T;
    g.L = L;
    g.M = r.M;
    g.kind = r.kind;
    g.inv_ref = r.inv_ref;
    g.tw_n1 = r.tw_n1;
    g.tw_M = r.tw_M;
    g.tw_b = r.tw_b;
    g.npass = 0;
    // stages: twiddles W_(ns R)^(rr k) by (rr - 1, block), the block's k being
    // its digits (earlier radices first) read least significant first
    std::vector<float2> tw(L);
    int ns = 1, at = 0;
    std::vector<int> off(r.nst), ns_of(r.nst);
    std::vector<int> k_of = {0};   // k of each block of the current stage
    for (int s = 0; s < r.nst; ++s) {
        const int R = r.radix[s];
        off[s] = at;
        ns_of[s] = ns;
        const int step = L / (ns * R);
        if (ns > 1)
            for (int rr = 1; rr < R; ++rr)
                for (int blk = 0; blk < ns; ++blk) {
                    const double ang = -2.0 * M_PI * static_cast<double>(rr * k_of[blk] * step) / L;
                    tw[at++] = make_float2(static_cast<float>(std::cos(ang)), static_cast<float>(std::sin(ang)));
                }
        std::vector<int> next(static_cast<size_t>(ns) * R);
        for (int blk = 0; blk < ns; ++blk)
            for (int k = 0; k < R; ++k) next[blk * R + k] = k_of[blk] + ns * k;
        k_of.swap(next);
        ns *= R;
    }
    std::vector<int> where(L);   // position of Z_k
    for (int q = 0; q < L; ++q) where[k_of[q]] = q;
    const int last = r.radix[r.nst - 1];
    g.pad = (last & 1) == 0 ? 1 : 0;
    g.zstride = g.pad ? L + (L + 15) / 16 : L;
    auto place = [&](int k) { return g.pad ? where[k] + (where[k] >> 4) : where[k]; };
    std::vector<int2> pos(T);
    for (int k = 0; k < T; ++k) {
        const int z = zidx[k];
        if (r.kind == CG_FFT_COSET)
            pos[k] = int2{place(z), 0};
        else
            pos[k] = int2{place(z == L ? 0 : z), place(z == 0 ? 0 : L - z)};
    }
    struct Cost {
        int per, cost;
    };
    std::vector<Cost> work;
    for (int s = 0; s < r.nst; ++s) {
        GenPass q{};
        q.ra = r.radix[s];
        q.rb = 1;
        q.ns = ns_of[s];
        q.off_a = off[s];
        if (s + 1 < r.nst && fusable(q.ra, r.radix[s + 1])) {
            q.rb = r.radix[s + 1];
            q.off_b = off[s + 1];
            ++s;
        }
        const int R = q.ra * q.rb;
        q.per = L / R;
        q.s = L / (q.ns * R);
        q.magic_per = magic_of(q.per);
        q.magic_s = magic_of(q.s);
        g.pass[g.npass++] = q;
        work.push_back({q.per, 15 + 14 * R});
    }
    if (r.kind == CG_FFT_COSET) work.push_back({L, 15 + 5 * r.M});
    work.push_back({T, 45});
    g.magic_l = magic_of(L);
    g.magic_t = magic_of(T);
    int o = align16(8 * L);
    g.sm_n1 = o;
    if (r.kind == CG_FFT_COSET) o = align16(o + 8 * (L + r.M));
    g.sm_b = o;
    if (r.kind != CG_FFT_COSET) o = align16(o + 8 * T);
    g.sm_pos = o;
    o = align16(o + 8 * T);
    g.sm_iref = o;
    o = align16(o + 4 * T);
    const int tables = o;
    cudaError_t e;
    void* fn = gen_ptr(g.pad != 0);
    if ((e = cudaMalloc(&p->d.gen_tw, sizeof(float2) * L)) != cudaSuccess) return e;
    if ((e = cudaMalloc(&p->d.gen_pos, sizeof(int2) * T)) != cudaSuccess) return e;
    if ((e = cudaMemcpy(p->d.gen_tw, tw.data(), sizeof(float2) * L, cudaMemcpyHostToDevice)) != cudaSuccess) return e;
    if ((e = cudaMemcpy(p->d.gen_pos, pos.data(), sizeof(int2) * T, cudaMemcpyHostToDevice)) != cudaSuccess) return e;
    g.tw = p->d.gen_tw;
    g.pos = p->d.gen_pos;
    // frames per block: least time per frame, counting the idle threads of the
    // passes' last rounds and the warps that fit an SM (six blocks by
    // registers; below about 20 warps latency shows)
    int smem_sm = 0, smem_block = 0;
    if ((e = cudaDeviceGetAttribute(&smem_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, p->device)) != cudaSuccess)
        return e;
    if ((e = cudaDeviceGetAttribute(&smem_block, cudaDevAttrMaxSharedMemoryPerBlockOptin, p->device)) != cudaSuccess)
        return e;
    double best = 0.0;
    for (int F = 1; F <= 32; ++F) {
        const int raw = tables, z = align16(raw + 2 * N * F + 32), total = align16(z + 8 * g.zstride * F);
        if (total > smem_block) break;
        const int blocks = std::min(6, smem_sm / (total + 1024));
        if (blocks < 1) break;
        double t = 0.0;
        for (const Cost& c : work) t += 60.0 + std::ceil(double(F) * c.per / kGenThreads) * c.cost;
        t = t / F / std::min(1.0, blocks * (kGenThreads / 32) / 20.0);
        if (best == 0.0 || t < best) {
            best = t;
            g.F = F;
            g.sm_raw = raw;
            g.sm_z = z;
            g.sm_total = total;
        }
    }
    if (best == 0.0) return cudaErrorInvalidValue;   // (the plan's own layout, which is larger, fitted)
    if ((e = raise_smem_limit(fn, g.sm_total)) != cudaSuccess) return e;
    int occ = 0;
    if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, fn, kGenThreads, g.sm_total)) != cudaSuccess) return e;
    p->grid_general = p->num_sms * std::max(occ, 1);
    return cudaSuccess;
}

cudaError_t launch_general_readout(const cg_plan_s* p, const int16_t* frames, int64_t n, float* amps, float* y,
                                   cudaStream_t s)
{
    GenArgs g = p->ga_gen;
    g.frames = frames;
    g.n_frames = n;
    g.amps = amps;
    g.y = y;
    // few frames: fewer per block, so that every SM has some
    const int64_t spread = (n + p->num_sms - 1) / p->num_sms;
    if (spread < g.F) g.F = static_cast<int>(spread);
    const int64_t nb = (n + g.F - 1) / g.F;
    const int grid = static_cast<int>(nb < p->grid_general ? nb : p->grid_general);
    void* args[] = {&g};
    return cudaLaunchKernel(gen_ptr(g.pad != 0), dim3(grid), dim3(kGenThreads), args, g.sm_total, s);
}

}  // namespace cg
