// Two-radix x pass with the k-space update (see evx_mixed.cuh).
#include <cfloat>

#include "evx_mixed.cuh"

namespace evx {
namespace mixed {

// a / D for D >= 1: the hardware's reciprocal and one Newton step on the quotient,
// q + r (a - D q), which rounds a result that is exact to about 2^-44 (a step on the
// reciprocal and a product by a round twice, the same way for a mode in every step).
// D = inf (|k|^4 beyond FP32) gives 0, as a division: the residual is taken at the largest
// finite number, inf * 0 would make the mode NaN and with it the field.
__device__ __forceinline__ float quotient(float a, float D) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(D));
    const float q = a * r;
    return fmaf(r, fmaf(-fminf(D, FLT_MAX), q, a), q);
}

// middle of the x pass: forward pass B of W and S, the update, inverse pass B;
// row k1 of the exchanges (column p). MODE as in XUpdArgs.model, 0 also for 1.
// SPILL: F_x W is put back into its own slots instead of being held in registers.
template <int MODE, bool SPILL>
struct ColUpdate {
    const XUpdArgs& a;
    float2* w;
    float2* s;
    const float* k2x;  // + k1
    int R1, k1;
    float k2yz, gpb;
    bool zero;  // row holds the k = 0 mode at k2 = 0
    __device__ __forceinline__ void blk(float k2, float Dinv, float& P, float& S) const {
        // P = L^n, S = sum_{j<n} L^j by binary powers: P_{2m} = P_m^2, S_{2m} = S_m (1 + P_m)
        const float Lk = fmaf(-a.dtM * k2, gpb, 1.f) * Dinv;
        P = 1.f, S = 0.f;
        for (int b = 31 - __clz(a.nblk); b >= 0; --b) {
            S = fmaf(S, P, S);
            P *= P;
            if ((a.nblk >> b) & 1) {
                S = fmaf(S, Lk, 1.f);
                P *= Lk;
            }
        }
    }
    template <int R>
    __device__ __forceinline__ void run() const {
        const bool ac = a.model == 1;
        float2 g[R];
#pragma unroll
        for (int i = 0; i < R; ++i) g[i] = w[i * CP];
        XDft<R, -1>::run(g);
        float2 v[R];
        if (MODE == 2) {  // preconditioner: dt / (1 + dt M kappa |k|^4) F_x W / L (dtM holds dt)
#pragma unroll
            for (int k = 0; k < R; ++k) {
                const float k2 = __ldg(k2x + R1 * k) + k2yz;
                v[k] = cscale(g[k], a.dtM * quotient(a.invL, fmaf(a.dtMk, k2 * k2, 1.f)));
            }
        } else {
            if (SPILL) {
#pragma unroll
                for (int i = 0; i < R; ++i) w[i * CP] = g[i];
            }
#pragma unroll
            for (int i = 0; i < R; ++i) v[i] = s[i * CP];
            XDft<R, -1>::run(v);
#pragma unroll
            for (int k = 0; k < R; ++k) {
                const float2 gk = SPILL ? w[k * CP] : g[k];
                const float k2 = __ldg(k2x + R1 * k) + k2yz;
                if (MODE == 3) {
                    const float Dinv = quotient(1.f, fmaf(a.dtMk, k2 * k2, 1.f));
                    float P, S;
                    blk(k2, Dinv, P, S);
                    const float bs = -a.dtM * k2 * Dinv * S * a.invL, as = P * a.invL;
                    v[k] = make_float2(fmaf(bs, gk.x, as * v[k].x), fmaf(bs, gk.y, as * v[k].y));
                } else {  // (c_hat - dt M |k|^2 g_hat) / (1 + dt M kappa |k|^4); Allen-Cahn: 1 and |k|^2
                    const float f = quotient(a.invL, fmaf(a.dtMk, ac ? k2 : k2 * k2, 1.f));
                    const float b = -a.dtM * (ac ? 1.f : k2);
                    v[k] = make_float2(f * fmaf(b, gk.x, v[k].x), f * fmaf(b, gk.y, v[k].y));
                }
            }
        }
        if (zero) v[0] = make_float2(0.f, 0.f);  // the mean is carried in FP64
        XDft<R, 1>::run(v);
        s[0] = v[0];
#pragma unroll
        for (int i = 1; i < R; ++i) s[i * CP] = twmul<1>(v[i], __ldg(a.tw + i * k1));
    }
};

// M1, M2: largest radices of R1 and R2
template <int MODE, int M1, int M2>
__global__ void __launch_bounds__(8 * M1, M1 <= 16 ? 5 : M1 <= 20 ? 4 : 2) mx_x_kernel(XUpdArgs a, int R1, int R2) {
    chain_wait();
    extern __shared__ float4 smem4[];
    const int p = threadIdx.x & 7, it = threadIdx.x >> 3, T = blockDim.x >> 3;
    const int R2p = R2 | 1, pitch = R2p * CP;
    float2* xw = reinterpret_cast<float2*>(smem4);
    float2* xs = MODE == 2 ? xw : xw + R1 * pitch;
    const int ky = blockIdx.y, kz = (int)blockIdx.x * CP + p;
    const bool valid = kz < a.ncols;
    const long long base = split_off(ky, a.YB, a.os, a.os2) + kz;
    const long long nbuf = (long long)(a.ny / a.YB) * a.os2;  // complex elements of W, S and S_out
    if (valid)
        for (int i = it; i < (MODE == 2 ? R2 : 2 * R2); i += T) {
            const bool second = i >= R2;
            const int n2 = second ? i - R2 : i;
            with_radix<M1>(R1, ColLoad<-1, XDft>{(second ? a.S : a.W) + base + n2 * a.rs, R2 * a.rs,
                                             (second ? xs : xw) + n2 * CP + p, pitch, a.tw, n2,
                                             {second ? a.S : a.W, nbuf}});
        }
    __syncthreads();
    if (valid) {
        const float k2yz = a.k2y[ky] + a.k2z[kz];
        const float gpb = MODE == 3 ? (float)(3.0 * (*a.cbar) * (*a.cbar) - 1.0) : 0.f;
        for (int k1 = it; k1 < R1; k1 += T)
            with_radix<M2>(R2, ColUpdate<MODE, (M2 > 16)>{a, xw + k1 * pitch + p, xs + k1 * pitch + p, a.k2x + k1, R1, k1,
                                                       k2yz, gpb, k1 == 0 && ky == 0 && kz == 0});
    }
    __syncthreads();
    if (valid)
        for (int n2 = it; n2 < R2; n2 += T)
            with_radix<M1>(R1, ColStoreInv{a.S_out + base + n2 * a.rs, R2 * a.rs, xs + n2 * CP + p, pitch, {a.S_out, nbuf}});
}

// gradient energy: forward passes A and B of S, sum of w(kz) |k|^2 |c_hat|^2 on FP32 pairs
struct ColEnergy {
    const float2* s;  // row k1
    const float* k2x;  // + k1
    int R1;
    double k2yz;
    bool edge;        // kz = 0 or M: weight 1, otherwise 2 (Hermitian half spectrum)
    double& acc;
    template <int R>
    __device__ __forceinline__ void run() const {
        float2 v[R];
#pragma unroll
        for (int i = 0; i < R; ++i) v[i] = s[i * CP];
        MxDft<R, -1>::run(v);
        PairSum ps;
        const float yh = (float)k2yz, yl = (float)(k2yz - (double)yh);
#pragma unroll
        for (int k = 0; k < R; ++k) {
            const float kx = __ldg(k2x + R1 * k);
            float2 k2 = two_sum(yh, kx);
            k2.y += yl;
            // pairs hold |c_hat|^2 and its product with |k|^2 while neither overflows and their low
            // parts (2^-48) stay normal numbers; anything else, NaN too, is added in FP64
            const float big = fmaxf(fabsf(v[k].x), fabsf(v[k].y)), e = big * big * k2.x;
            if (big != 0.f && !(big >= 0x1p-39f && big <= 0x1p50f && e >= 0x1p-78f && e <= 0x1p100f)) {
                acc += (edge ? 1.0 : 2.0) * ((double)kx + k2yz) * ((double)v[k].x * v[k].x + (double)v[k].y * v[k].y);
                continue;
            }
            const float px = v[k].x * v[k].x, py = v[k].y * v[k].y;
            float2 m = two_sum(px, py);
            m.y += fmaf(v[k].x, v[k].x, -px) + fmaf(v[k].y, v[k].y, -py);
            ps.add(mul22(k2, m));
        }
        acc += (edge ? 1.0 : 2.0) * ps.take();
    }
};
template <int MAX>
__global__ void __launch_bounds__(8 * MAX, MAX <= 16 ? 5 : 2) mx_energy_kernel(XEnergyArgs a, int R1, int R2) {
    chain_wait();
    extern __shared__ float4 smem4[];
    __shared__ double red[8];
    float2* xs = reinterpret_cast<float2*>(smem4);
    const int p = threadIdx.x & 7, it = threadIdx.x >> 3, T = blockDim.x >> 3;
    const int R2p = R2 | 1, pitch = R2p * CP;
    const int ky = blockIdx.y, kz = (int)blockIdx.x * CP + p;
    const bool valid = kz < a.ncols;
    const long long base = split_off(ky, a.YB, a.os, a.os2) + kz;
    const long long nbuf = (long long)(a.ny / a.YB) * a.os2;
    if (valid)
        for (int n2 = it; n2 < R2; n2 += T)
            with_radix<MAX>(R1, ColLoad<-1>{a.S + base + n2 * a.rs, R2 * a.rs, xs + n2 * CP + p, pitch, a.tw, n2, {a.S, nbuf}});
    __syncthreads();
    double acc = 0.0;
    if (valid) {
        const double k2yz = (double)a.k2y[ky] + (double)a.k2z[kz];
        for (int k1 = it; k1 < R1; k1 += T)
            with_radix<MAX>(R2, ColEnergy{xs + k1 * pitch + p, a.k2x + k1, R1, k2yz, kz == 0 || kz == a.M, acc});
    }
    // fixed-order sum of the CTA (its last warp may be partial)
    const int lane = threadIdx.x & 31, live = min(32, (int)blockDim.x - (int)(threadIdx.x & ~31));
    const unsigned here = live == 32 ? 0xffffffffu : (1u << live) - 1;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const double t = __shfl_down_sync(here, acc, o);
        if (lane + o < live) acc += t;
    }
    if (lane == 0) red[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < ((int)blockDim.x + 31) / 32; ++w) t += red[w];
        a.partials[(long long)blockIdx.y * gridDim.x + blockIdx.x] = t;
    }
}

}  // namespace mixed

int bounds_line_mixed_x(bool clear) { return EVX_BOUNDS_TAKE(clear); }

template <int MODE>
static auto mx_x_pick(int R1, int R2) {
    return R2 > 16   ? mixed::mx_x_kernel<MODE, 32, 32>
           : R1 > 20 ? mixed::mx_x_kernel<MODE, 32, 16>
           : R1 > 16 ? mixed::mx_x_kernel<MODE, 20, 16>
                     : mixed::mx_x_kernel<MODE, 16, 16>;
}

bool mixed_xupdate(const XUpdArgs& a, cudaStream_t st, cudaError_t* err) {
    int R1, R2;
    if (!a.W || !mixed_split(a.L, &R1, &R2)) return false;
    const size_t smem = sizeof(float2) * R1 * (R2 | 1) * SP * (a.model == 2 ? 1 : 2);
    auto kern = a.model == 3 ? mx_x_pick<3>(R1, R2) : a.model == 2 ? mx_x_pick<2>(R1, R2) : mx_x_pick<0>(R1, R2);
    if ((*err = mx_smem(kern, smem)) != cudaSuccess) return true;
    *err = launch_chained(kern, dim3(a.nchunks, a.ny), R1 * SP, smem, st, a, R1, R2);
    return true;
}

// The energy's x pass, of every length with two radices (the tuned kernels' among them:
// 313 us at 256^3 stage by stage with FP64 sums, 54 us now)
bool mixed_xenergy(const XEnergyArgs& a, cudaStream_t st, cudaError_t* err) {
    int R1, R2;
    if (!mixed_split(a.L, &R1, &R2)) return false;
    const size_t smem = sizeof(float2) * R1 * (R2 | 1) * SP;
    auto kern = R1 > 16 ? mixed::mx_energy_kernel<32> : mixed::mx_energy_kernel<16>;
    if ((*err = mx_smem(kern, smem)) != cudaSuccess) return true;
    *err = launch_chained(kern, dim3(a.nchunks, a.ny), R1 * SP, smem, st, a, R1, R2);
    return true;
}

}  // namespace evx
