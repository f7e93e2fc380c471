// Two-radix y pass (see evx_mixed.cuh).
#include "evx_mixed.cuh"

namespace evx {
namespace mixed {

template <int DIR, int MAX>
__global__ void __launch_bounds__(8 * MAX, MAX <= 16 ? 8 : MAX <= 20 ? 5 : 2) mx_y_kernel(SPassArgs a, int R1, int R2) {
    chain_wait();
    extern __shared__ float4 smem4[];
    float2* xb = reinterpret_cast<float2*>(smem4);
    const int p = threadIdx.x & 7, it = threadIdx.x >> 3, T = blockDim.x >> 3;
    const int R2p = R2 | 1;
    const bool valid = (int)blockIdx.x * CP + p < a.ncols;
    const long long base = (long long)blockIdx.y * a.os + (long long)blockIdx.x * CP + p;
    const long long nbuf = (long long)(a.L / a.YB) * a.os2;  // complex elements of in / out
    if (valid)
        for (int n2 = it; n2 < R2; n2 += T)
            with_radix<MAX>(R1, ColLoad<DIR>{a.in + base + n2 * a.rs, R2 * a.rs, xb + n2 * CP + p, R2p * CP, a.tw, n2, {a.in, nbuf}});
    __syncthreads();
    if (valid)
        for (int k1 = it; k1 < R1; k1 += T)
            with_radix<MAX>(R2, ColStore<DIR>{a.out + base + k1 * a.rs, R1 * a.rs, xb + k1 * R2p * CP + p, {a.out, nbuf}});
}

}  // namespace mixed

int bounds_line_mixed_y(bool clear) { return EVX_BOUNDS_TAKE(clear); }

// The radices of a length: the smallest R1 >= R2 whose product is L (0 if none).
bool mixed_split(int L, int* R1, int* R2) {
    static const int radices[] = {1, 2, 3, 4, 5, 6, 8, 9, 10, 12, 15, 16, 18, 20, 24, 25, 27, 30, 32};
    for (int r1 : radices) {
        if (L % r1) continue;
        const int r2 = L / r1;
        if (r2 > r1) continue;
        for (int r : radices)
            if (r == r2) {
                *R1 = r1;
                *R2 = r2;
                return true;
            }
    }
    return false;
}

// true if the strided rows can be addressed with one stride (plain layout)
static bool plain_rows(int YB, int ny) { return YB == ny; }

bool mixed_spass(const SPassArgs& a, int dir, cudaStream_t st, cudaError_t* err) {
    int R1, R2;
    if (!plain_rows(a.YB, a.L) || !mixed_split(a.L, &R1, &R2)) return false;
    const size_t smem = sizeof(float2) * R1 * (R2 | 1) * SP;
    auto kern = R1 > 20   ? (dir < 0 ? mixed::mx_y_kernel<-1, 32> : mixed::mx_y_kernel<1, 32>)
                : R1 > 16 ? (dir < 0 ? mixed::mx_y_kernel<-1, 20> : mixed::mx_y_kernel<1, 20>)
                          : (dir < 0 ? mixed::mx_y_kernel<-1, 16> : mixed::mx_y_kernel<1, 16>);
    if ((*err = mx_smem(kern, smem)) != cudaSuccess) return true;
    *err = launch_chained(kern, dim3(a.nchunks, a.nouter), R1 * SP, smem, st, a, R1, R2);
    return true;
}

}  // namespace evx
