// The mixed-radix passes of small grids with their stages grouped in registers:
// the arithmetic of the stage-by-stage kernels (evx_kernels.cu), operation for
// operation, in two register passes and one shared-memory exchange per transform
// instead of one exchange, two barriers and the index divisions per radix.
//
// A length L with the radix order r1, r2, ... (make_plan) is cut into a leading
// group R1 = r1 .. rm and a trailing group R2 = r(m+1) .. rn. The R1 elements
// n2 + R2 t (t < R1) are closed under the leading stages and the R2 elements
// k1 + R1 t under the trailing ones, so each group runs in one thread's registers:
// stage s of a group works on its R values as a Stockham stage of that length,
// with the twiddles exp(-2 pi i t kk / (Ns r)) of the whole transform.
//
// Why beside the two-radix kernels (evx_mixed.cuh), which need one exchange less
// per inverse and are faster: these give the fields of the stage-by-stage kernels
// to the bit, so data sets made with them (the surrogate trains on BF16
// activations, where a last-bit change of an input moves gradients by 1e-4) are
// reproduced. That is the only reason; it holds for the fields, not for the
// energies, and only up to STAGED_MAX_VOXELS. Measured on a GB300, microseconds per
// Cahn-Hilliard step (64 steps in a graph):
//   grid            stage by stage   grouped   two radices
//   24^3                  50.2         17.2        10.9
//   48 x 40 x 36          62.1         21.9        11.9
//   96^3                 158.8         78.7        17.4
//   120 x 108 x 100      174.9         60.0        22.4
//   300 x 120 x 108      382.2         69.0        49.1
// Per kernel at 48 x 40 x 36 (ncu, cold caches): stage by stage y 10.9, z 56, x 26
// us; grouped 4.7, 13.3, 23.4; two-radix 3.6, 8.0, 8.3.
#include <algorithm>
#include <cstdint>

#include "evx_cta_sum.cuh"
#include "evx_internal.h"

namespace evx {
namespace staged {

// leading radix of a group, as in make_plan: 5s, 3s, 16s, then 8, 4 or 2
__host__ __device__ constexpr int lead(int R) {
    return R % 5 == 0 ? 5 : R % 3 == 0 ? 3 : R % 16 == 0 ? 16 : R;
}

// the stages of a group of R values; NSI: product of the group's radices done.
// Ns, kk, L: of the whole transform at the group's start (L a multiple of Ns R)
template <int R, int NSI, int REST, int DIR>
__device__ __forceinline__ void stages(float2 (&v)[R], int Ns, int kk, int L, const float2* __restrict__ tw) {
    if constexpr (REST > 1) {
        constexpr int r = lead(REST);
        float2 o[R];
        const int tws = L / (Ns * NSI * r);
#pragma unroll
        for (int j = 0; j < R / r; ++j) {
            const int ki = j % NSI;
            float2 u[r];
#pragma unroll
            for (int t = 0; t < r; ++t) u[t] = v[j + t * (R / r)];
            if (Ns * NSI > 1) {
                const int step = tws * (kk + ki * Ns);
#pragma unroll
                for (int t = 1; t < r; ++t) {
                    float2 w = __ldg(tw + t * step);
                    if (DIR > 0) w.y = -w.y;
                    u[t] = cmul(u[t], w);
                }
            }
            Dft<r, DIR>::run(u);
#pragma unroll
            for (int t = 0; t < r; ++t) o[(j - ki) * r + ki + t * NSI] = u[t];
        }
#pragma unroll
        for (int i = 0; i < R; ++i) v[i] = o[i];
        stages<R, NSI * r, REST / r, DIR>(v, Ns, kk, L, tw);
    }
}
// group of one thread at Ns, kk
template <int R, int DIR>
__device__ __forceinline__ void group(float2 (&v)[R], int Ns, int kk, int L, const float2* tw) {
    stages<R, 1, R, DIR>(v, Ns, kk, L, tw);
}

#define EVX_STG_GROUPS(F) F(1) F(2) F(3) F(4) F(5) F(6) F(8) F(9) F(12) F(15) F(16) F(20) F(25) F(27) F(32)
template <typename Fn>
__device__ __forceinline__ void with_group(int r, Fn&& f) {
    switch (r) {
#define EVX_STG_CASE(R) \
    case R: f.template run<R>(); return;
        EVX_STG_GROUPS(EVX_STG_CASE)
#undef EVX_STG_CASE
        default: break;
    }
}

// ---------------------------------------------------------- y and x passes
// 8 adjacent columns per CTA; thread = (column p, item it). Slot of leading
// output k1 of item n2: (k1 R2p + n2) 8 + p, R2p = R2 | 1 (conflict-free both ways).
constexpr int CP = SP;

struct Cut {
    int L, R1, R2, R2p;
};

// leading group of column elements from global memory -> exchange
template <int DIR>
struct LeadFromGlobal {
    const float2* src;  // element n2
    long long stride;   // between elements R2 apart
    float2* x;          // exchange at (0, n2)
    Cut c;
    const float2* tw;
    Extent<float2> ext;
    template <int R>
    __device__ __forceinline__ void run() const {
        float2 v[R];
#pragma unroll
        for (int t = 0; t < R; ++t) v[t] = EVX_AT(src + t * stride, ext) ? src[t * stride] : make_float2(0.f, 0.f);
        group<R, DIR>(v, 1, 0, c.L, tw);
#pragma unroll
        for (int u = 0; u < R; ++u) x[u * c.R2p * CP] = v[u];
    }
};
// trailing group, row k1 of the exchange -> global elements k1 + R1 u
template <int DIR>
struct TrailToGlobal {
    const float2* x;  // exchange at (k1, 0)
    float2* dst;      // element k1
    long long stride;  // between elements R1 apart
    Cut c;
    const float2* tw;
    int k1;
    Extent<float2> ext;
    template <int R>
    __device__ __forceinline__ void run() const {
        float2 v[R];
#pragma unroll
        for (int t = 0; t < R; ++t) v[t] = x[t * CP];
        group<R, DIR>(v, c.R1, k1, c.L, tw);
#pragma unroll
        for (int u = 0; u < R; ++u)
            if (EVX_AT(dst + u * stride, ext)) dst[u * stride] = v[u];
    }
};

template <int DIR>
__global__ void __launch_bounds__(256, 3) stg_y_kernel(SPassArgs a, Cut c) {
    chain_wait();
    extern __shared__ float4 smem4[];
    float2* xb = reinterpret_cast<float2*>(smem4);
    const int p = threadIdx.x & 7, it = threadIdx.x >> 3;
    const bool valid = (int)blockIdx.x * CP + p < a.ncols;
    const long long base = (long long)blockIdx.y * a.os + (long long)blockIdx.x * CP + p;
    const long long nbuf = (long long)(c.L / a.YB) * a.os2;  // complex elements of in / out
    if (valid && it < c.R2)
        with_group(c.R1, LeadFromGlobal<DIR>{a.in + base + it * a.rs, c.R2 * a.rs, xb + it * CP + p, c, a.tw, {a.in, nbuf}});
    __syncthreads();
    if (valid && it < c.R1)
        with_group(c.R2, TrailToGlobal<DIR>{xb + it * c.R2p * CP + p, a.out + base + it * a.rs, c.R1 * a.rs, c, a.tw, it,
                                            {a.out, nbuf}});
}

// trailing groups of W and S, the update (the operations of xupdate_kernel), the
// new spectrum left in row k1 of S's exchange: element k1 + R1 u at slot u
struct UpdateRow {
    const XUpdArgs& a;
    const float2* w;
    float2* s;
    Cut c;
    int k1;
    float k2y, k2z, gpb;
    bool zero;
    template <int R>
    __device__ __forceinline__ void run() const {
        const bool pre = a.model == 2, blk = a.model == 3;
        float2 g[R], v[R];
#pragma unroll
        for (int t = 0; t < R; ++t) g[t] = w[t * CP];
        group<R, -1>(g, c.R1, k1, c.L, a.tw);
        if (!pre) {
#pragma unroll
            for (int t = 0; t < R; ++t) v[t] = s[t * CP];
            group<R, -1>(v, c.R1, k1, c.L, a.tw);
        } else {
#pragma unroll
            for (int t = 0; t < R; ++t) v[t] = make_float2(0.f, 0.f);
        }
#pragma unroll
        for (int u = 0; u < R; ++u) {
            const float k2 = __ldg(a.k2x + k1 + c.R1 * u) + k2y + k2z;
            const float ainv = a.invL / fmaf(a.dtMk, a.model == 1 ? k2 : k2 * k2, 1.f);
            const float b = -a.dtM * (a.model == 1 ? 1.f : k2) * ainv;
            const float2 ch = v[u], gh = g[u];
            float2 r = make_float2(ainv * ch.x, ainv * ch.y);
            if (blk) {
                const float Lk = fmaf(-a.dtM * k2, gpb, 1.f) * ainv * (float)c.L;
                float P = 1.f, S = 0.f;
                for (int j = 0; j < a.nblk; ++j) {
                    S += P;
                    P *= Lk;
                }
                const float bs = -a.dtM * k2 * ainv * S;
                r = make_float2(fmaf(bs, gh.x, P * a.invL * ch.x), fmaf(bs, gh.y, P * a.invL * ch.y));
            } else if (pre) {
                r = make_float2(a.dtM * ainv * gh.x, a.dtM * ainv * gh.y);
            } else {
                r.x = fmaf(b, gh.x, r.x);
                r.y = fmaf(b, gh.y, r.y);
            }
            if (zero && u == 0) r = make_float2(0.f, 0.f);
            v[u] = r;
        }
#pragma unroll
        for (int u = 0; u < R; ++u) s[u * CP] = v[u];
    }
};
// leading group of the inverse: elements n2 + R2 t of the spectrum left in rows
// (element k at slot (k mod R1) R2p + k / R1) -> exchange x. DIST: distance of
// neighbouring slots. SYNC: the two may be the same buffer.
template <int DIR, int DIST, bool SYNC>
struct LeadFromRows {
    const float2* rows;
    float2* x;  // exchange at (0, n2)
    Cut c;
    const float2* tw;
    int n2;
    bool act;
    template <int R>
    __device__ __forceinline__ void run() const {
        float2 v[R];
        if (act) {
            int q = n2 / c.R1, m = n2 - q * c.R1;
            const int dq = c.R2 / c.R1, dm = c.R2 - dq * c.R1;
#pragma unroll
            for (int t = 0; t < R; ++t) {
                v[t] = rows[(m * c.R2p + q) * DIST];
                q += dq;
                m += dm;
                if (m >= c.R1) {
                    m -= c.R1;
                    ++q;
                }
            }
        }
        if (SYNC) __syncthreads();
        if (act) {
            group<R, DIR>(v, 1, 0, c.L, tw);
#pragma unroll
            for (int u = 0; u < R; ++u) x[u * c.R2p * DIST] = v[u];
        }
    }
};

__global__ void __launch_bounds__(256, 2) stg_x_kernel(XUpdArgs a, Cut c) {
    chain_wait();
    extern __shared__ float4 smem4[];
    const int p = threadIdx.x & 7, it = threadIdx.x >> 3;
    const int ky = blockIdx.y, kz = (int)blockIdx.x * CP + p;
    const bool valid = kz < a.ncols;
    float2* xw = reinterpret_cast<float2*>(smem4);
    float2* xs = xw + c.R1 * c.R2p * CP;
    const long long base = split_off(ky, a.YB, a.os, a.os2) + kz;
    const long long nbuf = (long long)(a.ny / a.YB) * a.os2;  // complex elements of W, S and S_out
    if (valid && it < c.R2) {
        with_group(c.R1, LeadFromGlobal<-1>{a.W + base + it * a.rs, c.R2 * a.rs, xw + it * CP + p, c, a.tw, {a.W, nbuf}});
        if (a.model != 2)
            with_group(c.R1, LeadFromGlobal<-1>{a.S + base + it * a.rs, c.R2 * a.rs, xs + it * CP + p, c, a.tw, {a.S, nbuf}});
    }
    __syncthreads();
    if (valid && it < c.R1) {
        const float gpb = a.model == 3 ? (float)(3.0 * (*a.cbar) * (*a.cbar) - 1.0) : 0.f;
        with_group(c.R2, UpdateRow{a, xw + it * c.R2p * CP + p, xs + it * c.R2p * CP + p, c, it, a.k2y[ky], a.k2z[kz], gpb,
                                   it == 0 && ky == 0 && kz == 0});
    }
    __syncthreads();
    if (valid && it < c.R2)
        with_group(c.R1, LeadFromRows<1, CP, false>{xs + p, xw + it * CP + p, c, a.tw, it, true});
    __syncthreads();
    if (valid && it < c.R1)
        with_group(c.R2, TrailToGlobal<1>{xw + it * c.R2p * CP + p, a.S_out + base + it * a.rs, c.R1 * a.rs, c, a.tw, it,
                                          {a.S_out, nbuf}});
}

// ---------------------------------------------------------------- z passes
// blockDim = (T, rows), T = max(R1, R2); a row of RS slots per thread row.
// C2R pre-processing and the inverse's leading group
struct PreLead {
    float2* row;
    Cut c;
    const float2* tw;
    const float2* rtw;
    int n2;
    bool act;
    template <int R>
    __device__ __forceinline__ void run() const {
        float2 v[R];
        if (act) {
#pragma unroll
            for (int t = 0; t < R; ++t) {
                const int k = n2 + c.R2 * t;
                const float2 xk = row[k], xm = row[c.L - k];
                if (k == 0) {
                    v[t] = make_float2(xk.x + xm.x, xk.x - xm.x);
                } else {
                    const float2 A = make_float2(xk.x + xm.x, xk.y - xm.y);
                    const float2 B = make_float2(xk.x - xm.x, xk.y + xm.y);
                    v[t] = cadd(A, mul_i<1>(cmul(cconj(__ldg(rtw + k)), B)));
                }
            }
        }
        __syncthreads();
        if (act) {
            group<R, 1>(v, 1, 0, c.L, tw);
#pragma unroll
            for (int u = 0; u < R; ++u) row[u * c.R2p + n2] = v[u];
        }
    }
};
// trailing group of the inverse and the pointwise stage; real samples k1 + R1 u stay in row k1
template <int MODE>
struct TrailPoint {
    float2* x;
    const ZPassArgs& a;
    Cut c;
    int k1;
    long long row;
    float cb, cbl, gp, c3;
    float& gs;
    float& ge;
    template <int R>
    __device__ __forceinline__ void run() const {
        float2 v[R];
#pragma unroll
        for (int t = 0; t < R; ++t) v[t] = x[t];
        group<R, 1>(v, c.R1, k1, c.L, a.tw);
        const float s = a.scale;
#pragma unroll
        for (int u = 0; u < R; ++u) {
            const int n = k1 + c.R1 * u;
            const float2 z = v[u];
            if (MODE == Z_ADJ) {
                const float2 cn = EVX_IN(row * a.cnpitch + 2 * n + 1, a.nrows * a.cnpitch)
                                      ? reinterpret_cast<const float2*>(a.cn + row * a.cnpitch)[n]
                                      : make_float2(0.f, 0.f);
                const float d0 = fmaf(3.f * cn.x, cn.x, -1.f), d1 = fmaf(3.f * cn.y, cn.y, -1.f);
                x[u] = make_float2(z.x * s * d0, z.y * s * d1);
                continue;
            }
            const float c0 = fmaf(z.x, s, cbl) + cb, c1 = fmaf(z.y, s, cbl) + cb;
            if (MODE == Z_C2R) {
                x[u] = make_float2(c0, c1);
                continue;
            }
            if (a.rout && EVX_IN(row * a.rpitch + 2 * n + 1, a.nrows * a.rpitch))
                reinterpret_cast<float2*>(a.rout + row * a.rpitch)[n] = make_float2(c0, c1);
            const float d0 = z.x * s, d1 = z.y * s;
            const float2 gv = make_float2(d0 * fmaf(d0, c3 + d0, gp), d1 * fmaf(d1, c3 + d1, gp));
            x[u] = gv;
            if (a.gsum) {
#pragma unroll
                for (int q = 0; q < 2; ++q) {  // TwoSum: the FP32 sum and its error term
                    const float val = q ? gv.y : gv.x, t = gs + val, bp = t - gs;
                    ge += (gs - (t - bp)) + (val - bp);
                    gs = t;
                }
            }
        }
    }
};
// trailing group of the forward transform -> Z_k in natural order
struct TrailNatural {
    float2* row;
    Cut c;
    const float2* tw;
    int k1;
    bool act;
    template <int R>
    __device__ __forceinline__ void run() const {
        float2 v[R];
        if (act) {
#pragma unroll
            for (int t = 0; t < R; ++t) v[t] = row[k1 * c.R2p + t];
            group<R, -1>(v, c.R1, k1, c.L, tw);
        }
        __syncthreads();
        if (act) {
#pragma unroll
            for (int u = 0; u < R; ++u) row[k1 + c.R1 * u] = v[u];
        }
    }
};
// leading group of the forward transform from a natural-order row
struct LeadNatural {
    float2* row;
    Cut c;
    const float2* tw;
    float cb, cbl;
    int n2;
    bool act;
    template <int R>
    __device__ __forceinline__ void run() const {
        float2 v[R];
        if (act) {
#pragma unroll
            for (int t = 0; t < R; ++t) {
                const float2 x = row[n2 + c.R2 * t];
                v[t] = make_float2((x.x - cb) - cbl, (x.y - cb) - cbl);
            }
        }
        __syncthreads();
        if (act) {
            group<R, -1>(v, 1, 0, c.L, tw);
#pragma unroll
            for (int u = 0; u < R; ++u) row[u * c.R2p + n2] = v[u];
        }
    }
};

template <int MODE>
__global__ void __launch_bounds__(256, 2) stg_z_kernel(ZPassArgs a, Cut c, int RS) {
    chain_wait();
    extern __shared__ float4 smem4[];
    float2* buf = reinterpret_cast<float2*>(smem4);
    __shared__ double red[256];
    const int tx = threadIdx.x, ty = threadIdx.y, T = blockDim.x, M = a.M;
    const int tid = ty * T + tx, nthr = T * blockDim.y;
    const long long row = (long long)blockIdx.x * blockDim.y + ty;
    const bool rowok = row < a.nrows;
    float2* z = buf + ty * RS;
    const double cbd = a.cbar ? *a.cbar : 0.0;
    const float cb = (float)cbd, cbl = (float)(cbd - (double)cb);
    const long long ur = MODE == Z_R2C || MODE == Z_C2R ? (a.map_rows ? user_row(rowok ? row : 0, a.YB, a.nxr, a.nyr) : row) : 0;
    if (rowok) {
        if (MODE == Z_R2C) {
            const float2* src = reinterpret_cast<const float2*>(a.rin + ur * a.rpitch);
            for (int n = tx; n < M; n += T)
                z[n] = EVX_IN(ur * a.rpitch + 2 * n + 1, a.nrows * a.rpitch) ? src[n] : make_float2(0.f, 0.f);
        } else {
            const float2* src = a.in + row * a.Zp;
            for (int n = tx; n <= M; n += T) z[n] = EVX_IN(row * a.Zp + n, a.nrows * a.Zp) ? src[n] : make_float2(0.f, 0.f);
        }
    }
    __syncthreads();
    const bool lead = rowok && tx < c.R2, trail = rowok && tx < c.R1;
    float gs = 0.f, ge = 0.f;
    if (MODE == Z_R2C) {
        with_group(c.R1, LeadNatural{z, c, a.tw, cb, cbl, tx, lead});
    } else {
        with_group(c.R1, PreLead{z, c, a.tw, a.rtw, tx, lead});
        __syncthreads();
        const float gp = a.nl_only ? 0.f : (float)(3.0 * cbd * cbd - 1.0), c3 = (float)(3.0 * cbd);
        if (trail) with_group(c.R2, TrailPoint<MODE>{z + tx * c.R2p, a, c, tx, row, cb, cbl, gp, c3, gs, ge});
        __syncthreads();
        if (MODE == Z_C2R) {
            double acc = 0.0;
            PairSum ps;
            if (rowok) {
                float2* o = a.partials ? nullptr : reinterpret_cast<float2*>(a.rout + ur * a.rpitch);
                for (int n = tx; n < M; n += T) {
                    const int q = n / c.R1, m = n - q * c.R1;
                    float2 v = z[m * c.R2p + q];
                    if (a.partials) {  // energy: nothing is written
                        add_well(ps, acc, v.x);
                        add_well(ps, acc, v.y);
                    } else if (!EVX_IN(ur * a.rpitch + 2 * n + 1, a.nrows * a.rpitch)) {
                    } else if (a.accumulate) {
                        const float2 prev = o[n];
                        o[n] = make_float2(prev.x + v.x, prev.y + v.y);
                    } else {
                        o[n] = v;
                    }
                }
            }
            if (a.partials) {
                red[tid] = acc + ps.take();
                __syncthreads();
                if (tid < 32) {
                    const double t = first_warp_sum(red, nthr, tid);
                    if (tid == 0) a.partials[blockIdx.x] = t;
                }
            }
            return;
        }
        with_group(c.R1, LeadFromRows<-1, 1, true>{z, z + tx, c, a.tw, tx, lead});
    }
    __syncthreads();
    with_group(c.R2, TrailNatural{z, c, a.tw, tx, trail});
    __syncthreads();
    if (rowok) {  // R2C post-processing
        float2* out = a.out + row * a.Zp;
        for (int k = tx; k <= M; k += T) {
            if (!EVX_IN(row * a.Zp + k, a.nrows * a.Zp)) continue;
            if (k == 0 || k == M) {
                const float2 z0 = z[0];
                out[k] = make_float2(k == 0 ? z0.x + z0.y : z0.x - z0.y, 0.f);
            } else {
                const float2 zk = z[k], zm = z[M - k];
                const float2 A = make_float2(0.5f * (zk.x + zm.x), 0.5f * (zk.y - zm.y));
                const float2 B = make_float2(0.5f * (zk.x - zm.x), 0.5f * (zk.y + zm.y));
                out[k] = cadd(A, mul_i<-1>(cmul(__ldg(a.rtw + k), B)));
            }
        }
    }
    if (MODE == Z_STEP && a.gsum) {
        red[tid] = (double)gs + (double)ge;
        __syncthreads();
        if (tid < 32) {
            const double t = first_warp_sum(red, nthr, tid);
            if (tid == 0) a.gsum[blockIdx.x] = t;
        }
    }
}

}  // namespace staged

// ----------------------------------------------------------------- dispatch
int bounds_line_staged(bool clear) { return EVX_BOUNDS_TAKE(clear); }

// The cut of a plan with both groups compiled in and the fewest threads per
// pencil; lengths up to 128 (longer ones have none or run better on two radices).
static bool staged_cut(const Plan& pl, int L, staged::Cut* c) {
    auto known = [](int r) {
#define EVX_STG_KNOWN(R) \
    if (r == R) return true;
        EVX_STG_GROUPS(EVX_STG_KNOWN)
#undef EVX_STG_KNOWN
        return false;
    };
    if (L > 128) return false;
    int best = 0, r1 = 1;
    for (int s = 0; s < pl.n; ++s) {
        r1 *= pl.r[s];
        const int r2 = L / r1, t = std::max(r1, r2);
        if (known(r1) && known(r2) && (!best || t < best)) {
            best = t;
            *c = staged::Cut{L, r1, r2, r2 | 1};
        }
    }
    return best > 0;
}

bool staged_spass(const SPassArgs& a, int dir, cudaStream_t st, cudaError_t* err) {
    staged::Cut c;
    if (!a.small || a.YB != a.L || !staged_cut(a.plan, a.L, &c)) return false;
    const size_t smem = sizeof(float2) * c.R1 * c.R2p * SP;  // at most 128 x 33 / 32 rows of 64 B: 9 KB
    auto kern = dir < 0 ? staged::stg_y_kernel<-1> : staged::stg_y_kernel<1>;
    *err = launch_chained(kern, dim3(a.nchunks, a.nouter), std::max(c.R1, c.R2) * SP, smem, st, a, c);
    return true;
}

bool staged_xupdate(const XUpdArgs& a, cudaStream_t st, cudaError_t* err) {
    staged::Cut c;
    if (!a.small || !a.W || !staged_cut(a.plan, a.L, &c)) return false;
    const size_t smem = 2 * sizeof(float2) * c.R1 * c.R2p * SP;
    *err = launch_chained(staged::stg_x_kernel, dim3(a.nchunks, a.ny), std::max(c.R1, c.R2) * SP, smem, st, a, c);
    return true;
}

// rows per CTA: up to 256 threads, fewer while the launch would leave SMs idle
static int staged_zrows(const ZPassArgs& a, const staged::Cut& c, int RS) {
    const int T = std::max(c.R1, c.R2);
    int rpc = std::max(1, std::min(256 / T, (int)(40 * 1024 / (sizeof(float2) * RS))));
    while (rpc > 1 && rpc * T > 32 && a.nrows / rpc < 2 * 152) rpc = (rpc + 1) / 2;
    return rpc;
}
static int staged_zstride(const ZPassArgs& a, const staged::Cut& c) {
    return std::max(a.M + 1, c.R1 * c.R2p) | 1;  // odd: the rows of a warp start on different banks
}
int staged_zgrid(const ZPassArgs& a) {
    staged::Cut c;
    if (!a.small || !staged_cut(a.plan, a.M, &c)) return 0;
    const int rpc = staged_zrows(a, c, staged_zstride(a, c));
    return (int)((a.nrows + rpc - 1) / rpc);
}

bool staged_zpass(const ZPassArgs& a, int mode, cudaStream_t st, cudaError_t* err, int* grid_used) {
    staged::Cut c;
    if (!a.small || !staged_cut(a.plan, a.M, &c)) return false;
    const float* real = mode == Z_R2C ? a.rin : mode == Z_ADJ ? a.cn : a.rout;
    const long long pitch = mode == Z_ADJ ? a.cnpitch : a.rpitch;
    if (real && (((uintptr_t)real & 7) || (pitch & 1))) return false;
    if (mode == Z_C2R && !a.rout && !a.partials) return false;
    const int RS = staged_zstride(a, c), rpc = staged_zrows(a, c, RS), T = std::max(c.R1, c.R2);
    const int grid = (int)((a.nrows + rpc - 1) / rpc);
    auto kern = mode == Z_STEP  ? staged::stg_z_kernel<Z_STEP>
                : mode == Z_ADJ ? staged::stg_z_kernel<Z_ADJ>
                : mode == Z_R2C ? staged::stg_z_kernel<Z_R2C>
                                : staged::stg_z_kernel<Z_C2R>;
    if (grid_used) *grid_used = grid;
    *err = launch_chained(kern, grid, dim3(T, rpc), sizeof(float2) * RS * rpc, st, a, c, RS);
    return true;
}

}  // namespace evx
