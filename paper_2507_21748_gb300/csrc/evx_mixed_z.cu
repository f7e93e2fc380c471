// Two-radix z passes (see evx_mixed.cuh).
#include "evx_cta_sum.cuh"
#include "evx_mixed.cuh"

namespace evx {
namespace mixed {

// ---------------------------------------------------------------- z passes
// A CTA holds RPC = blockDim.y rows of RS slots; thread (tx, ty) works on row ty,
// items tx < R2 or R1 (T = blockDim.x = R1 >= R2). Rows enter and leave in
// natural order; slot (k1, n2) of the exchange is k1 R2p + n2. tA[k1 R2 + n2] and
// tB[n2 R1 + k1] hold w_M^{n2 k1} in the order the lanes read it.
__device__ __forceinline__ void cp16(void* smem, const void* g) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"((unsigned)__cvta_generic_to_shared(smem)), "l"(g)
                 : "memory");
}
__device__ __forceinline__ void cp8(void* smem, const void* g) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"((unsigned)__cvta_generic_to_shared(smem)), "l"(g)
                 : "memory");
}
__device__ __forceinline__ void cp_wait_all() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }

struct ZRow {
    float2* row;  // this row's slots
    int R1, R2, R2p, M;
    const float2* tA;
    const float2* tB;
    const float2* rtw;
};

// C2R pre-processing and inverse pass A: the row (natural order) -> exchange
struct ZInvA {
    ZRow z;
    int n2;
    bool act;
    template <int R>
    __device__ __forceinline__ void run() const {
        float2 v[R];
        if (act) {
#pragma unroll
            for (int i = 0; i < R; ++i) {
                const int k = n2 + z.R2 * i;
                float2 xk = z.row[k], xm = z.row[z.M - k];
                if (k == 0) xk.y = xm.y = 0.f;  // a real field's k = 0 and Nyquist values are real
                const float2 w = __ldg(z.rtw + k);
                const float px = xk.x + xm.x, py = xk.y - xm.y, qx = xk.x - xm.x, qy = xk.y + xm.y;
                v[i] = make_float2(fmaf(-w.x, qy, fmaf(w.y, qx, px)), fmaf(w.x, qx, fmaf(w.y, qy, py)));
            }
        }
        __syncthreads();  // rows read: their slots become the exchange
        if (act) {
            MxDft<R, 1>::run(v);
            z.row[n2] = v[0];
#pragma unroll
            for (int k = 1; k < R; ++k) z.row[k * z.R2p + n2] = twmul<1>(v[k], __ldg(z.tA + k * z.R2 + n2));
        }
    }
};
// inverse pass B, the pointwise stage, forward pass B, in row k1 of the exchange
template <bool ADJ>
struct ZMiddle {
    ZRow z;
    const ZPassArgs& a;
    int k1;
    long long row;
    bool rowok;
    float cb, cbl, gp, c3;
    float& gs;  // sum of the stage's values (Allen-Cahn) and the sum of its rounding errors
    float& ge;
    template <int R>
    __device__ __forceinline__ void run() const {
        float2* x = z.row + k1 * z.R2p;
        float2 v[R];
#pragma unroll
        for (int i = 0; i < R; ++i) v[i] = x[i];
        MxDft<R, 1>::run(v);
        const float s = a.scale;
#pragma unroll
        for (int k = 0; k < R; ++k) {
            const int m = k1 + z.R1 * k;
            const float d0 = v[k].x * s, d1 = v[k].y * s;
            if (ADJ) {
                const float2 c = rowok && EVX_IN(row * a.cnpitch + 2 * m + 1, a.nrows * a.cnpitch)
                                     ? reinterpret_cast<const float2*>(a.cn + row * a.cnpitch)[m]
                                     : make_float2(0.f, 0.f);
                v[k] = make_float2(d0 * fmaf(3.f * c.x, c.x, -1.f), d1 * fmaf(3.f * c.y, c.y, -1.f));
            } else {
                if (a.rout && rowok && EVX_IN(row * a.rpitch + 2 * m + 1, a.nrows * a.rpitch))
                    reinterpret_cast<float2*>(a.rout + row * a.rpitch)[m] =
                        make_float2(fmaf(v[k].x, s, cbl) + cb, fmaf(v[k].y, s, cbl) + cb);
                // g(c) - g(cbar) about the mean, as in the fast z pass
                v[k] = make_float2(d0 * fmaf(d0, c3 + d0, gp), d1 * fmaf(d1, c3 + d1, gp));
                if (a.gsum && rowok) {
#pragma unroll
                    for (int q = 0; q < 2; ++q) {  // TwoSum: the FP32 sum and its error term
                        const float val = q ? v[k].y : v[k].x, t = gs + val, bp = t - gs;
                        ge += (gs - (t - bp)) + (val - bp);
                        gs = t;
                    }
                }
            }
        }
        MxDft<R, -1>::run(v);
        x[0] = v[0];
#pragma unroll
        for (int i = 1; i < R; ++i) x[i] = twmul<-1>(v[i], __ldg(z.tB + i * z.R1 + k1));
    }
};
// inverse pass B to the real row c = z / (ny nz) + cbar in natural order (shared memory)
struct ZInvB {
    ZRow z;
    float s, cb, cbl;
    int k1;
    bool act;
    template <int R>
    __device__ __forceinline__ void run() const {
        float2 v[R];
        if (act) {
            const float2* x = z.row + k1 * z.R2p;
#pragma unroll
            for (int i = 0; i < R; ++i) v[i] = x[i];
            MxDft<R, 1>::run(v);
        }
        __syncthreads();
        if (act) {
#pragma unroll
            for (int k = 0; k < R; ++k)
                z.row[k1 + z.R1 * k] = make_float2(fmaf(v[k].x, s, cbl) + cb, fmaf(v[k].y, s, cbl) + cb);
        }
    }
};
// forward pass B from a real row in natural order (minus the mean hi + lo)
struct ZFwdB {
    ZRow z;
    float hi, lo;
    int k1;
    bool act;
    template <int R>
    __device__ __forceinline__ void run() const {
        float2 v[R];
        if (act) {
#pragma unroll
            for (int k = 0; k < R; ++k) {
                const float2 c = z.row[k1 + z.R1 * k];
                v[k] = make_float2((c.x - hi) - lo, (c.y - hi) - lo);
            }
        }
        __syncthreads();
        if (act) {
            MxDft<R, -1>::run(v);
            float2* x = z.row + k1 * z.R2p;
            x[0] = v[0];
#pragma unroll
            for (int i = 1; i < R; ++i) x[i] = twmul<-1>(v[i], __ldg(z.tB + i * z.R1 + k1));
        }
    }
};
// forward pass A: column n2 of the exchange -> Z_k in natural order
struct ZFwdA {
    ZRow z;
    int n2;
    bool act;
    template <int R>
    __device__ __forceinline__ void run() const {
        float2 v[R];
        if (act) {
#pragma unroll
            for (int k = 0; k < R; ++k) v[k] = z.row[k * z.R2p + n2];
        }
        __syncthreads();
        if (act) {
            MxDft<R, -1>::run(v);
#pragma unroll
            for (int i = 0; i < R; ++i) z.row[n2 + z.R2 * i] = v[i];
        }
    }
};

template <int MODE, int MAX>
__global__ void __launch_bounds__(MAX > 16 ? 256 : 192, MAX > 16 ? 2 : MAX > 12 ? 3 : 4) mx_z_kernel(ZPassArgs a, int R1, int R2, int RS) {
    chain_wait();
    extern __shared__ float4 smem4[];
    float2* buf = reinterpret_cast<float2*>(smem4);
    const int tx = threadIdx.x, ty = threadIdx.y, T = blockDim.x, RPC = blockDim.y, M = a.M;
    const int tid = ty * T + tx, nthr = T * RPC;
    const long long row0 = (long long)blockIdx.x * RPC, row = row0 + ty;
    const int nr = (int)min((long long)RPC, a.nrows - row0);
    const bool rowok = ty < nr;
    const double cbd = a.cbar ? *a.cbar : 0.0;
    const float cb = (float)cbd, cbl = (float)(cbd - (double)cb);
    ZRow z{buf + ty * RS, R1, R2, R2 | 1, M, a.twA, a.twA + M, a.rtw};
    // rows into shared memory, a row to a thread row
    if (MODE == Z_R2C) {
        if (rowok) {
            const long long ur = a.map_rows ? user_row(row, a.YB, a.nxr, a.nyr) : row;
            const float2* src = reinterpret_cast<const float2*>(a.rin + ur * a.rpitch);
            for (int q = tx; q < M; q += T)
                if (EVX_IN(ur * a.rpitch + 2 * q + 1, a.nrows * a.rpitch)) cp8(z.row + q, src + q);
        }
    } else if (rowok) {
        const float2* src = a.in + row * a.Zp;
        for (int q = tx; q < a.Zp / 2; q += T)
            if (EVX_IN(row * a.Zp + 2 * q + 1, a.nrows * a.Zp)) cp16(z.row + 2 * q, src + 2 * q);
    }
    cp_wait_all();
    __syncthreads();
    const bool actA = rowok && tx < R2, actB = rowok;  // T = R1
    float gs = 0.f, ge = 0.f;
    if (MODE == Z_R2C) {
        with_radix<MAX>(R2, ZFwdB{z, cb, cbl, tx, actB});
        __syncthreads();
    } else {
        with_radix<MAX>(R1, ZInvA{z, tx, actA});
        __syncthreads();
        if (MODE == Z_C2R) {
            with_radix<MAX>(R2, ZInvB{z, a.scale, cb, cbl, tx, actB});
            __syncthreads();
            if (a.partials) {  // energy: nothing is written
                double acc = 0.0;
                PairSum ps;
                if (rowok)
                    for (int q = tx; q < M; q += T) {
                        add_well(ps, acc, z.row[q].x);
                        add_well(ps, acc, z.row[q].y);
                    }
                __shared__ double red[256];
                red[tid] = acc + ps.take();
                __syncthreads();
                if (tid < 32) {
                    const double t = first_warp_sum(red, nthr, tid);
                    if (tid == 0) a.partials[blockIdx.x] = t;
                }
                return;
            }
            if (rowok) {
                const long long ur = a.map_rows ? user_row(row, a.YB, a.nxr, a.nyr) : row;
                float2* dst = reinterpret_cast<float2*>(a.rout + ur * a.rpitch);
                auto ok = [&](int q) { return EVX_IN(ur * a.rpitch + 2 * q + 1, a.nrows * a.rpitch); };
                if (a.accumulate) {  // eight reads in flight
                    for (int q = tx; q < M; q += 8 * T) {
                        float2 prev[8];
#pragma unroll
                        for (int u = 0; u < 8; ++u)
                            if (q + u * T < M) prev[u] = ok(q + u * T) ? dst[q + u * T] : make_float2(0.f, 0.f);
#pragma unroll
                        for (int u = 0; u < 8; ++u)
                            if (q + u * T < M && ok(q + u * T)) dst[q + u * T] = cadd(prev[u], z.row[q + u * T]);
                    }
                } else {
                    for (int q = tx; q < M; q += T)
                        if (ok(q)) dst[q] = z.row[q];
                }
            }
            return;
        }
        const float gp = a.nl_only ? 0.f : (float)(3.0 * cbd * cbd - 1.0), c3 = (float)(3.0 * cbd);
        if (actB) with_radix<MAX>(R2, ZMiddle<MODE == Z_ADJ>{z, a, tx, row, rowok, cb, cbl, gp, c3, gs, ge});
        __syncthreads();
    }
    with_radix<MAX>(R1, ZFwdA{z, tx, actA});
    __syncthreads();
    // R2C post-processing, pairs (k, M - k)
    if (rowok) {
        float2* out = a.out + row * a.Zp;
        auto put = [&](int k, float2 v) {
            if (EVX_IN(row * a.Zp + k, a.nrows * a.Zp)) out[k] = v;
        };
        for (int k = tx; k <= M / 2; k += T) {
            if (k == 0) {
                const float2 z0 = z.row[0];
                put(0, make_float2(z0.x + z0.y, 0.f));
                put(M, make_float2(z0.x - z0.y, 0.f));
                continue;
            }
            // X_k = (P - i w Q) / 2, P = Z_k + conj Z_{M-k}, Q = Z_k - conj Z_{M-k}; X_{M-k} = conj(P + i w Q) / 2
            const float2 zk = z.row[k], zm = z.row[M - k], w = __ldg(z.rtw + k);
            const float px = 0.5f * (zk.x + zm.x), py = 0.5f * (zk.y - zm.y);
            const float qx = 0.5f * (zk.x - zm.x), qy = 0.5f * (zk.y + zm.y);
            const float ux = fmaf(w.x, qy, w.y * qx), uy = fmaf(-w.x, qx, w.y * qy);  // -i w Q
            put(k, make_float2(px + ux, py + uy));
            if (M - k != k) put(M - k, make_float2(px - ux, uy - py));
        }
    }
    if (MODE == Z_STEP && a.gsum) {  // FP64 partial of the CTA, fixed order
        __shared__ double red[256];
        red[tid] = (double)gs + (double)ge;
        __syncthreads();
        if (tid < 32) {
            const double t = first_warp_sum(red, nthr, tid);
            if (tid == 0) a.gsum[blockIdx.x] = t;
        }
    }
}

}  // namespace mixed

int bounds_line_mixed_z(bool clear) { return EVX_BOUNDS_TAKE(clear); }

// rows per CTA: up to 192 threads (256 with radices above 16) and 48 KB, fewer while the grid would leave SMs idle
static int mixed_zrows(const ZPassArgs& a, int R1, int RS) {
    int rpc = std::max(1, std::min((R1 > 16 ? 256 : 192) / R1, (int)(48 * 1024 / (sizeof(float2) * RS))));
    while (rpc > 1 && rpc * R1 > 32 && a.nrows / rpc < 2 * 152) rpc = (rpc + 1) / 2;
    return rpc;
}
static int mixed_zstride(const ZPassArgs& a, int R1, int R2) {
    const int rs = std::max(a.Zp, R1 * (R2 | 1));
    const int want = (R1 + 1) & ~1;  // = T (mod 16), even (16-byte copies)
    return rs + (((want - rs) % 16) + 16) % 16;
}

int mixed_zgrid(const ZPassArgs& a) {
    int R1, R2;
    if (!a.twA || !mixed_split(a.M, &R1, &R2)) return 0;
    const int rpc = mixed_zrows(a, R1, mixed_zstride(a, R1, R2));
    return (int)((a.nrows + rpc - 1) / rpc);
}

bool mixed_zpass(const ZPassArgs& a, int mode, cudaStream_t st, cudaError_t* err, int* grid_used) {
    int R1, R2;
    if (!a.twA || !mixed_split(a.M, &R1, &R2)) return false;
    const float* real = mode == Z_R2C ? a.rin : mode == Z_ADJ ? a.cn : a.rout;
    const long long pitch = mode == Z_ADJ ? a.cnpitch : a.rpitch;
    if (real && (((uintptr_t)real & 7) || (pitch & 1))) return false;
    if (mode == Z_C2R && !a.rout && !a.partials) return false;
    const int RS = mixed_zstride(a, R1, R2), rpc = mixed_zrows(a, R1, RS);
    const int grid = (int)((a.nrows + rpc - 1) / rpc);
    const size_t smem = sizeof(float2) * RS * rpc;
    auto pick = [&](auto small, auto mid, auto big) { return R1 > 16 ? big : R1 > 12 ? mid : small; };
    void (*kern)(ZPassArgs, int, int, int) = nullptr;
#define EVX_MX_Z(MODE) \
    case MODE: kern = pick(mixed::mx_z_kernel<MODE, 12>, mixed::mx_z_kernel<MODE, 16>, mixed::mx_z_kernel<MODE, 32>); break;
    switch (mode) {
        EVX_MX_Z(Z_STEP)
        EVX_MX_Z(Z_ADJ)
        EVX_MX_Z(Z_R2C)
        EVX_MX_Z(Z_C2R)
        default: return false;
    }
#undef EVX_MX_Z
    if ((*err = mx_smem(kern, smem)) != cudaSuccess) return true;
    if (grid_used) *grid_used = grid;
    *err = launch_chained(kern, grid, dim3(R1, rpc), smem, st, a, R1, R2, RS);
    return true;
}

}  // namespace evx
