// Two-radix passes for every other 2/3/5-smooth length L = R1 R2 (R1, R2 <= 32):
// the y pass, the x pass with the k-space update, the z passes.
//
// Four-step FFT of a length-L pencil, n = n2 + R2 n1, k = k1 + R1 k2:
//   pass A: item n2 (R2 of them): DFT-R1 over n1 in registers, times w_L^{n2 k1}
//   pass B: item k1 (R1 of them): DFT-R2 over n2 in registers
// One shared-memory exchange between the two, and none elsewhere: pass A of the
// y and x passes reads its R1 values straight from global memory (8 adjacent
// columns = 64-byte rows, R1 independent loads in flight per thread) and the
// last pass writes straight back. The radices are compile-time (register DFTs),
// which ones a launch uses is a uniform switch, so a handful of kernels serve
// all lengths; a stage-by-stage Stockham kernel pays one exchange, two barriers
// and the index divisions per radix (evx_kernels.cu, kept for lengths that are
// no product of two radices up to 32: 972 and 1000).
//
// The exchange keeps item k1's R2 values in a row of R2p = R2 | 1 slots: pass A
// writes neighbouring slots, pass B reads an odd distance apart, both without
// bank conflicts. Every thread rewrites only the slots it has read, so an
// inverse walks back through the same slots with one barrier per exchange.
//
// Measured on a GB300 against the stage-by-stage kernels, 300 x 240 x 200: y pass
// 137 -> 21 us (5.5 TB/s), z pass 237 -> 55 us, x pass 620 -> 62 us; 48 x 40 x 36:
// y 10.9 -> 3.6, z 56 -> 8, x 26 -> 8 us. The y pass is bound by memory, the z and
// x passes by instruction issue and their barriers.
#pragma once
#include <algorithm>
#include <cstdint>

#include "evx_internal.h"

namespace evx {
namespace mixed {

// ------------------------------------------------------------------ radices
#define EVX_MX_RADICES(F) \
    F(1) F(2) F(3) F(4) F(5) F(6) F(8) F(9) F(10) F(12) F(15) F(16) F(18) F(20) F(24) F(25) F(27) F(30) F(32)

// f.template run<R>() for the radix r <= MAX. Kernels are compiled for a few MAX: the
// registers of a kernel are those of its largest radix.
template <int MAX, typename Fn>
__device__ __forceinline__ void with_radix(int r, Fn&& f) {
    switch (r) {
#define EVX_MX_CASE(R)                                 \
    case R:                                            \
        if constexpr (R <= MAX) f.template run<R>();   \
        return;
        EVX_MX_RADICES(EVX_MX_CASE)
#undef EVX_MX_CASE
        default: break;
    }
}

// The register DFTs of these passes. 10 and 20 from coprime factors, without twiddles: the
// rounded twiddles of the forms the four-step kernels use scale a transform and its inverse
// by a fixed amount, and the state goes through both along x in every step (a length of 300:
// 1 + 4.0e-8 against 1 + 2.4e-8 this way; the radices 5 5 4 3 one by one 1 + 2.2e-8).
template <int R, int DIR> struct MxDft : Dft<R, DIR> {};
template <int DIR> struct MxDft<10, DIR> : DftCoprime<2, 5, DIR> {};
template <int DIR> struct MxDft<20, DIR> : DftCoprime<4, 5, DIR> {};

// Along x, radices with several factors of 3 take sin(2 pi / 3) as a sum of two floats: its
// rounding (-1.8e-8) shrinks a transform and its inverse by up to 3.6e-8 per factor, for some
// modes in every step (with the rounded constant the field after 20 steps on 864 x 40 x 60 was
// 17%, on 324 x 40 x 60 10% further from 64 bits than stage by stage; 9% and 19% closer this
// way). A single factor of 3 keeps it: next to factors of 5, whose constants err the other
// way, it helps. So do the y and z passes, which the state does not go through every step.
template <int R, int DIR> struct FineDft : Dft<R, DIR> {};
template <int DIR>
struct FineDft<3, DIR> {
    __device__ __forceinline__ static void run(float2* v) {
        constexpr double H = 0.86602540378443864676;  // sin(2 pi / 3)
        constexpr float hi = (float)H, lo = (float)(H - (double)hi);
        const float2 t = cadd(v[1], v[2]), s = csub(v[1], v[2]);
        const float2 m = make_float2(fmaf(-0.5f, t.x, v[0].x), fmaf(-0.5f, t.y, v[0].y));
        const float2 r = mul_i<DIR>(make_float2(fmaf(s.x, hi, s.x * lo), fmaf(s.y, hi, s.y * lo)));
        v[0] = cadd(v[0], t);
        v[1] = cadd(m, r);
        v[2] = csub(m, r);
    }
};
template <int DIR> struct FineDft<9, DIR> : DftTwiddled<3, 3, DIR, FineDft> {};
template <int R, int DIR> struct XDft : MxDft<R, DIR> {};
template <int DIR> struct XDft<9, DIR> : FineDft<9, DIR> {};
template <int DIR> struct XDft<18, DIR> : DftCoprime<2, 9, DIR, FineDft> {};
template <int DIR> struct XDft<27, DIR> : DftTwiddled<3, 9, DIR, FineDft> {};

template <int DIR>
__device__ __forceinline__ float2 twmul(float2 v, float2 w) {
    if (DIR > 0) w.y = -w.y;
    return cmul(v, w);
}

// ------------------------------------------- column tiles (x and y passes)
// A CTA holds SP = 8 adjacent columns; thread = (p, it), p = column, items it,
// it + T, ... Slot of (k1, n2): (k1 R2p + n2) 8 + p.
constexpr int CP = SP;

// pass A from global: v[n1] = src[n1 stride], DFT-R1, twiddle, into column n2 of the exchange
template <int DIR, template <int, int> class F = MxDft>
struct ColLoad {
    const float2* src;
    long long stride;
    float2* x;  // exchange, at column p and n2
    int pitch;  // R2p * 8
    const float2* tw;
    int n2;
    Extent<float2> ext;
    template <int R>
    __device__ __forceinline__ void run() const {
        float2 v[R];
#pragma unroll
        for (int i = 0; i < R; ++i) v[i] = EVX_AT(src + i * stride, ext) ? src[i * stride] : make_float2(0.f, 0.f);
        F<R, DIR>::run(v);
        x[0] = v[0];
#pragma unroll
        for (int k = 1; k < R; ++k) x[k * pitch] = twmul<DIR>(v[k], __ldg(tw + n2 * k));
    }
};
// pass B to global: v[n2] from row k1 of the exchange, DFT-R2, dst[k2 stride]
template <int DIR>
struct ColStore {
    float2* dst;
    long long stride;
    const float2* x;  // exchange, at column p and row k1
    Extent<float2> ext;
    template <int R>
    __device__ __forceinline__ void run() const {
        float2 v[R];
#pragma unroll
        for (int i = 0; i < R; ++i) v[i] = x[i * CP];
        MxDft<R, DIR>::run(v);
#pragma unroll
        for (int k = 0; k < R; ++k)
            if (EVX_AT(dst + k * stride, ext)) dst[k * stride] = v[k];
    }
};
// last pass of an inverse, to global: v[k1] from column n2, DFT-R1, dst[n1 stride]
struct ColStoreInv {
    float2* dst;
    long long stride;
    const float2* x;  // exchange, at column p and n2
    int pitch;
    Extent<float2> ext;
    template <int R>
    __device__ __forceinline__ void run() const {
        float2 v[R];
#pragma unroll
        for (int k = 0; k < R; ++k) v[k] = x[k * pitch];
        XDft<R, 1>::run(v);
#pragma unroll
        for (int i = 0; i < R; ++i)
            if (EVX_AT(dst + i * stride, ext)) dst[i * stride] = v[i];
    }
};

}  // namespace mixed

template <typename K>
static cudaError_t mx_smem(K kernel, size_t bytes) {
    if (bytes <= 48 * 1024) return cudaSuccess;
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

}  // namespace evx
