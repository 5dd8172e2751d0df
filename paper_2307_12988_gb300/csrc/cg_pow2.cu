// cg_pow2.cu -- tooth readout for frames whose teeth share no residue class
// (the full real transform) when N = 2 L with L = 1024, 2048 or 4096.
//
// Paper ("Data Capture and Processing"): each row of N samples is Fourier
// transformed and the tooth bins are read.  The real row is packed as L
// complex values z_n = x_{2n} + i x_{2n+1}; the L-point DFT is factored as
// L = 16 x 16 x R3 (R3 = L / 256) and run in three register passes with
// compile-time sizes, L / 16 threads per frame and 16 values per thread:
//   pass 1  n = n1 + (L/16) n2:  DFT16 over n2 -> k2, twiddle W_L^{n1 k2};
//   pass 2  n1 = m1 + R3 m2:     DFT16 over m2 -> j,  twiddle W_{L/16}^{m1 j};
//   pass 3                        DFT_R3 over m1 -> j',
// so that Z[k2 + 16 j + 256 j'] = sum_n z_n W_L^{n k}.  The passes work in
// place: a thread writes its results where it read its points, so after pass 1
// the points of a warp's butterflies are its own (k2 blocks of L / 16) and
// passes 2 and 3 need no barrier but the warp's.  The real-FFT split
// X_b = E + W_N^b O is evaluated only at the teeth.  The samples go straight
// from global memory to the registers of pass 1, one frame ahead.
//
// What bounds it: the shared-memory pipe (68 % busy: 870 wavefronts of 128
// bytes a 4,096-sample frame) and instruction issue (55 %).  So the twiddles
// of pass 1, which a thread needs unchanged in every frame, live in its
// registers, and so do the next frame's samples: 128 registers, 512 threads an
// SM.  30,000 frames of 4,096 samples, 201 teeth: 163 us with samples staged
// and three barriered exchanges through shared memory, 150 in place at 768
// threads with the twiddles in shared memory, 123 so.
#include <cstdint>
#include <cuda_runtime.h>

#include "cg_fft.cuh"
#include "cg_internal.h"
#include "cg_tc.cuh"

namespace cg {

namespace {

template <int L>
struct Pow2Plan {
    static constexpr int TPF = L / 16;             // threads per frame
    static constexpr int NTH = TPF > 128 ? TPF : 128;   // threads per block
    static constexpr int FPB = NTH / TPF;          // frames in flight per block
    static constexpr int R3 = L / 256;
    static constexpr int PP = 16 / R3;             // pass-3 butterflies per thread
    static constexpr int N = 2 * L;
};

// Place of point p: its low four bits XORed with the next four, which puts the
// points of every access of a half warp on distinct banks (strides 1, R3 and
// L / 16).  Linear over XOR: p ^ d with d disjoint from p is reached from the
// address of p by a constant XOR and a constant offset.
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

template <int L>
__global__ void __launch_bounds__(Pow2Plan<L>::NTH, 512 / Pow2Plan<L>::NTH) pow2_readout_kernel(ReadoutArgs a)
{
    using P = Pow2Plan<L>;
    constexpr int TPF = P::TPF, FPB = P::FPB, R3 = P::R3, PP = P::PP, N = P::N;
    extern __shared__ __align__(1024) unsigned char sm[];
    tc::pdl_start();
    const int T = a.T;
    float2* Z = reinterpret_cast<float2*>(sm);                         // [FPB][L]
    // pass twiddles laid out so a warp reads consecutive entries:
    // tw1[k2][n1] = W_L^{n1 k2}, tw2[j][m1] = W_{L/16}^{m1 j}
    float2* tw2 = Z + FPB * L;                                         // [16][R3]
    float2* twb = tw2 + 16 * R3;                                       // [T] W_N^{b_k}
    int2* pos = reinterpret_cast<int2*>(twb + T);                      // [T] places of Z_b and Z_(L - b)
    float* iref = reinterpret_cast<float*>(pos + T);                   // [T]
    const int fs = threadIdx.x / TPF;      // frame slot
    const int lt = threadIdx.x % TPF;      // thread within the frame
    const int lane = threadIdx.x & 31;
    const int64_t step = static_cast<int64_t>(gridDim.x) * FPB;
    int64_t f = static_cast<int64_t>(blockIdx.x) * FPB + fs;
    uint32_t next[16];                     // the next frame's samples, two a word
    auto fetch = [&](int64_t fr) {
        const uint32_t* rw = reinterpret_cast<const uint32_t*>(a.frames + fr * N) + lt;
#pragma unroll
        for (int n2 = 0; n2 < 16; ++n2) next[n2] = __ldcs(rw + TPF * n2);
    };
    if (f < a.n_frames) fetch(f);
    float2 tw1[16];                        // W_L^{n1 k2} of the thread's n1 = lt
#pragma unroll
    for (int k2 = 1; k2 < 16; ++k2) tw1[k2] = a.tw_L[lt * k2];
    for (int i = threadIdx.x; i < 16 * R3; i += P::NTH) {
        const int j = i / R3, m1 = i - j * R3;
        tw2[i] = a.tw_L[16 * m1 * j];
    }
    // place of Z_k: k = k2 + 16 j + 256 j' lies at point k2 L/16 + R3 j + j'
    auto place = [](int k) { return zsw((k & 15) * TPF + ((k >> 4) & 15) * R3 + (k >> 8)); };
    for (int i = threadIdx.x; i < T; i += P::NTH) {
        const int b = a.zidx[i];
        twb[i] = a.tw_b[i];
        pos[i] = make_int2(place(b == L ? 0 : b), place(b == 0 ? 0 : L - b));
        iref[i] = a.inv_ref[i];
    }
    __syncthreads();
    const float2* Zf = Z + fs * L;
    const uint32_t z = static_cast<uint32_t>(__cvta_generic_to_shared(Zf));
    const uint32_t z1 = z + 8 * zsw(lt);                                  // pass 1: points lt + TPF n2
    const uint32_t z2 = z + 8 * zsw((lt / R3) * TPF + lt % R3);           // pass 2: (k2, m1), points R3 m2 on
    // pass 3: butterflies (k2, j) of the warp's own k2 blocks, 16 a block
    const int k2w = (lt >> 5) * (32 / R3);
    auto group_sync = [&] {
        asm volatile("bar.sync %0, %1;\n" ::"r"(fs + 1), "n"(TPF) : "memory");
    };
    for (; f < a.n_frames; f += step) {
        // ---- pass 1: DFT16 over n2, twiddle W_L^{n1 k2} ----
        {
            float2 v[16];
#pragma unroll
            for (int n2 = 0; n2 < 16; ++n2)
                v[n2] = make_float2(static_cast<float>(static_cast<short>(next[n2] & 0xffffu)),
                                    static_cast<float>(static_cast<short>(next[n2] >> 16)));
            if (f + step < a.n_frames) fetch(f + step);
            Dft<16>::run(v);
#pragma unroll
            for (int k2 = 1; k2 < 16; ++k2) v[k2] = cmul(v[k2], tw1[k2]);
#pragma unroll
            for (int k2 = 0; k2 < 16; ++k2) zst(zat(z1, k2 * TPF), v[k2]);
        }
        group_sync();
        // ---- pass 2: DFT16 over m2, twiddle W_{L/16}^{m1 j} ----
        {
            float2 v[16];
#pragma unroll
            for (int m2 = 0; m2 < 16; ++m2) v[m2] = zld(zat(z2, R3 * m2));
            Dft<16>::run(v);
#pragma unroll
            for (int j = 1; j < 16; ++j) v[j] = cmul(v[j], tw2[j * R3 + lt % R3]);
#pragma unroll
            for (int j = 0; j < 16; ++j) zst(zat(z2, R3 * j), v[j]);
        }
        __syncwarp();
        // ---- pass 3: DFT_R3 over m1 ----
#pragma unroll
        for (int i = 0; i < PP; ++i) {
            const int q = lane + 32 * i;
            const uint32_t z3 = z + 8 * zsw((k2w + (q >> 4)) * TPF + R3 * (q & 15));
            float2 v[R3];
#pragma unroll
            for (int m1 = 0; m1 < R3; ++m1) v[m1] = zld(zat(z3, m1));
            Dft<R3>::run(v);
#pragma unroll
            for (int m1 = 0; m1 < R3; ++m1) zst(zat(z3, m1), v[m1]);
        }
        group_sync();
        // ---- teeth: real-FFT split at the tooth bins, coalesced outputs ----
        const int64_t row = f * T;
        for (int k = lt; k < T; k += TPF) {
            const int2 p = pos[k];
            const float2 Zb = Zf[p.x];
            const float2 Zr = Zf[p.y];
            // E = (Zb + conj Zr) / 2, O = (Zb - conj Zr) / (2 i), X_b = E + W_N^b O
            const float2 E = make_float2(0.5f * (Zb.x + Zr.x), 0.5f * (Zb.y - Zr.y));
            const float2 Dd = make_float2(0.5f * (Zb.x - Zr.x), 0.5f * (Zb.y + Zr.y));
            const float2 O = make_float2(Dd.y, -Dd.x);
            const float2 X = cadd(E, cmul(twb[k], O));
            const float amp = cabs_approx(X);
            if (a.amps) a.amps[row + k] = amp;
            if (a.y) a.y[row + k] = __fmul_rn(amp, iref[k]);
        }
        group_sync();   // the teeth are read before the next frame's points land
    }
}

template <int L>
void* pow2_fn()
{
    return reinterpret_cast<void*>(&pow2_readout_kernel<L>);
}

void* pow2_ptr(int L)
{
    switch (L) {
    case 1024: return pow2_fn<1024>();
    case 2048: return pow2_fn<2048>();
    case 4096: return pow2_fn<4096>();
    default: return nullptr;
    }
}

int pow2_threads(int L) { return L / 16 > 128 ? L / 16 : 128; }
int pow2_fpb(int L) { return pow2_threads(L) / (L / 16); }

}  // namespace

// Chooses the power-of-two readout for full real transforms with L = N / 2 in
// {1024, 2048, 4096}: shared memory (the frames' points, twiddles and tooth
// tables) and the grid; leaves pow2_ok false
// otherwise.
cudaError_t setup_pow2(cg_plan_s* p)
{
    p->pow2_ok = false;
    if (p->kind != CG_FFT_FULL || p->M != 2) return cudaSuccess;
    const int L = p->L, T = p->T;
    void* fn = pow2_ptr(L);
    if (!fn) return cudaSuccess;
    const int fpb = pow2_fpb(L);
    ReadoutArgs& r = p->pa;
    r = p->ra;
    r.sm_total = 8 * (fpb * L + 16 * (L / 256) + 2 * T) + 4 * T;
    cudaError_t e;
    if ((e = raise_smem_limit(fn, r.sm_total)) != cudaSuccess) return e;
    int occ = 0;
    if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, fn, pow2_threads(L), r.sm_total)) != cudaSuccess)
        return e;
    if (occ < 1) return cudaSuccess;
    p->grid_pow2 = p->num_sms * occ;
    p->pow2_ok = true;
    return cudaSuccess;
}

cudaError_t launch_pow2_readout(const cg_plan_s* p, const int16_t* frames, int64_t n, float* amps, float* y,
                                cudaStream_t s)
{
    ReadoutArgs r = p->pa;
    r.frames = frames;
    r.n_frames = n;
    r.amps = amps;
    r.y = y;
    const int fpb = pow2_fpb(p->L);
    const int64_t nb = (n + fpb - 1) / fpb;
    const int grid = static_cast<int>(nb < p->grid_pow2 ? nb : p->grid_pow2);
    void* args[] = {&r};
    return cudaLaunchKernel(pow2_ptr(p->L), dim3(grid), dim3(pow2_threads(p->L)), args, r.sm_total, s);
}

}  // namespace cg
