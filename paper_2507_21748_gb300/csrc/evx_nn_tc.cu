// tcgen05 engine of the surrogate's 32 -> 32 convolutions (sm_103a).
//
// conv_ring_kernel computes the periodic 3x3x3 convolution as an implicit GEMM on
// the 5th-generation tensor cores: D[128 voxels x N] (FP32, in tensor memory)
// += A[128 x 16] (BF16 activations, shared memory) x B[16 x N] (BF16 weights,
// shared memory), over the taps and 2 K-steps of 16 input channels. The
// weights use the no-swizzle K-major core-matrix layout (a core matrix is
// 8 rows x 16 bytes stored as 128 contiguous bytes; the descriptor gives the
// distance of core matrices adjacent along K (leading byte offset, 128 B) and
// along N (stride byte offset, 512 B)).
//
// It is a persistent, warp-specialised pipeline. A work unit is a run of output rows (b, x, y = ys .. ye-1,
// z0 .. z0+127); the 128 voxels of a row are the MMA's M. The kernel walks the
// INPUT rows y' = ys-1 .. ye: a ring slot holds input row (b, x-1 .. x+1, y')
// as [dx][z][32 ci] with 64-byte z rows in the 64-byte swizzle layout, exactly
// as TMA writes it (row 16 + i holds z0 + i, rows 0..15 and 144..159 the
// periodic halo), so the operand of tap dz starts dz rows later and its second
// K-step 32 bytes on. One input row feeds output rows y'+1, y', y'-1 (dy = -1,
// 0, +1): the weights of the three dy are stacked along N = 96, so each input
// row costs 18 MMAs (3 dx x 3 dz x 2 K-steps) into three consecutive
// accumulator blocks of a 16-block ring (32 columns per output row, descending
// with the row so that the three blocks are adjacent; where they wrap past
// column 511 each MMA splits into N = 64 + 32). Blocks start at zero and only
// accumulate; an output row is complete after its third input row.
//   warp 0      producer: per slot 9 TMA loads (per dx the 128 rows z0 ..
//               and two 16-row halo boxes at (z0-16) mod Z, (z0+128) mod Z);
//               a full mbarrier per slot; a slot is refilled once the
//               commit of the row it held (below) has fired
//   warp 1      MMA issuer: the warp walks the schedule converged; lane 0 waits,
//               issues (predicated, not branched) and commits once per input
//               row, on the block of the output row that row completes (which
//               also frees the row's slot)
//   warps 2..9  epilogue: each warp reads 16 columns of its 32 lanes of a
//               completed block (tcgen05.ld), zeroes them (tcgen05.st), frees
//               the block, applies bias and the fused epilogue and stores BF16
//               channels-last; the two partial rows at each end of a unit are
//               dropped
// Rows are walked along y when Z is a multiple of 128 and along x otherwise: an
// output's taps are then added in the order (dy, dx, dz) and (dx, dy, dz), the
// orders earlier versions used for these sizes (results to the bit).
//
// When Z is an odd multiple of 64 the last z chunk of a row holds 64 voxels: the
// producer loads 64-row boxes, the MMAs still run with M = 128 (the upper lanes
// accumulate stale rows, and are zeroed and not stored). Half of such a chunk's
// tensor work is idle, but an unpipelined kernel with 2 x 64 voxel tiles took
// 740 us where this takes 170 us (4 x 64^3, GELU epilogue).
//
// Every mbarrier wait is bounded (about 1 s); a wait that runs out sets the
// device flag g_tc_timeout, makes the other roles stop, waits (bounded) for
// its own copies and MMAs in flight, frees the tensor memory and returns. The
// host reads the flag with tc_take_timeout.
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "../../include/evx_nn.h"
#include "evx_nn_common.cuh"

namespace evxnn {

__device__ int g_tc_timeout;

// ------------------------------------------------------------- primitives
__device__ __forceinline__ uint64_t sdesc(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
    uint64_t d = 0;
    d |= (uint64_t)((saddr >> 4) & 0x3FFF);
    d |= (uint64_t)((lbo >> 4) & 0x3FFF) << 16;
    d |= (uint64_t)((sbo >> 4) & 0x3FFF) << 32;
    d |= (uint64_t)1 << 46;  // descriptor version (sm_100 family); no swizzle, base offset 0
    return d;
}

// K-major operand in the 64-byte swizzle layout (rows of 64 bytes, 16-byte
// chunks permuted by address bits 7..8 within 512-byte atoms): rows 64 bytes
// apart, 8-row groups 512 bytes apart. The permutation follows the absolute
// shared-memory address (as TMA applies it), so a start moved by whole rows
// or by 32 bytes addresses the same stored layout.
__device__ __forceinline__ uint64_t sdesc_sw64(uint32_t saddr) { return sdesc(saddr, 16, 512) | (4ull << 61); }

// instruction descriptor, kind::f16: D FP32, A and B BF16, both K-major, N, M
__host__ __device__ constexpr uint32_t idesc_bf16(int M, int N) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

// one MMA, executed by the whole (converged) warp and issued by lane 0 alone
// through an instruction predicate: no divergent branch around the issue, which
// on sm_103a took the ring's 18-MMA issue sequence from about 1,570 to 1,200 cycles
__device__ __forceinline__ void tc_mma_lane0(uint32_t dtmem, uint64_t a, uint64_t b, uint32_t idesc) {
    asm volatile(
        "{\n .reg .pred p, q;\n .reg .u32 l;\n mov.u32 l, %%laneid;\n setp.eq.u32 p, l, 0;\n"
        " setp.ne.b32 q, %4, 0;\n @p tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, q;\n}\n" ::"r"(dtmem),
        "l"(a), "l"(b), "r"(idesc), "r"(1)
        : "memory");
}

// arrive on bar once every MMA this thread issued before has completed
__device__ __forceinline__ void tc_commit(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar)
                 : "memory");
}

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        " selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}

// bounded wait (about 2 s) for the phase of the given parity
__device__ __forceinline__ bool tc_wait(uint32_t bar, uint32_t parity) {
    const long long t0 = clock64();
    while (true) {
        if (mbar_try(bar, parity)) return true;
        if (clock64() - t0 > (1LL << 32)) return false;
    }
}

__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}

__device__ __forceinline__ void tma_load4(uint32_t dst, const CUtensorMap* map, int c0, int c1, int c2, int c3,
                                          uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], "
        "[%6];" ::"r"(dst),
        "l"(map), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(bar)
        : "memory");
}

__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&r)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr)
        : "memory");
}

__device__ __forceinline__ void fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// bias + fused epilogue on NCH (a multiple of 8) channels c0 .. of voxel vox,
// r = FP32 accumulator bits, bias = the NCH biases (registers), pf = the voxel's
// pre-activations (GELU_BWD), loaded ahead; BF16 stores of 16 bytes
template <int EPI, int NCH>
__device__ __forceinline__ void epilogue_store(const ConvArgs& a, long long vox, int c0, const uint32_t* r,
                                               const float* bias, const uint4* pf) {
    const long long o = vox * 32 + c0;
#pragma unroll
    for (int q = 0; q < NCH / 8; ++q) {
        float v[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) v[j] = __uint_as_float(r[q * 8 + j]) + bias[q * 8 + j];
        uint4 outw;
        __nv_bfloat162* ow = reinterpret_cast<__nv_bfloat162*>(&outw);
        if (EPI == EVX_NN_EPI_GELU) {
            uint4 pw;
            __nv_bfloat162* pp = reinterpret_cast<__nv_bfloat162*>(&pw);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                pp[j] = __floats2bfloat162_rn(v[2 * j], v[2 * j + 1]);
                ow[j] = __floats2bfloat162_rn(gelu(v[2 * j]), gelu(v[2 * j + 1]));
            }
            if (a.pre) *reinterpret_cast<uint4*>(a.pre + o + q * 8) = pw;  // NULL: inference, not kept
        } else if (EPI == EVX_NN_EPI_GELU_BWD) {
            const uint4 pw = pf[q];
            const __nv_bfloat162* pp = reinterpret_cast<const __nv_bfloat162*>(&pw);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const float2 pf = __bfloat1622float2(pp[j]);
                ow[j] = __floats2bfloat162_rn(v[2 * j] * gelu_grad(pf.x), v[2 * j + 1] * gelu_grad(pf.y));
            }
        } else if (EPI == EVX_NN_EPI_RESID) {
            const uint4 rw = *reinterpret_cast<const uint4*>(a.res + o + q * 8);
            const __nv_bfloat162* rp = reinterpret_cast<const __nv_bfloat162*>(&rw);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const float2 rf = __bfloat1622float2(rp[j]);
                ow[j] = __floats2bfloat162_rn(v[2 * j] + rf.x, v[2 * j + 1] + rf.y);
            }
        } else {
#pragma unroll
            for (int j = 0; j < 4; ++j) ow[j] = __floats2bfloat162_rn(v[2 * j], v[2 * j + 1]);
        }
        *reinterpret_cast<uint4*>(reinterpret_cast<__nv_bfloat16*>(a.out) + o + q * 8) = outw;
    }
}

// EVX_NN_EPI_RESID32 for one epilogue warp: 32 voxels vox0 .. vox0 + 31 (lane = voxel
// of acc) x 16 channels c0 ... The sums are staged in shared memory ([voxel][16],
// 16-byte chunk c of row v at chunk c ^ ((v >> 1) & 3): conflict-free both ways) and
// the stream is read and written with lane l on voxel l / 4 + 8 i, channels
// c0 + 4 (l % 4) ..: every instruction covers 8 whole 64-byte row pieces instead of
// one 16-byte piece of 32 rows. s: the stream's values, loaded ahead by resid32_load.
__device__ __forceinline__ void resid32_load(const ConvArgs& a, long long vox0, int c0, int lane, float4 (&s)[4]) {
#pragma unroll
    for (int i = 0; i < 4; ++i)
        s[i] = *reinterpret_cast<const float4*>(reinterpret_cast<const float*>(a.pre) +
                                                (vox0 + (lane >> 2) + 8 * i) * 32 + c0 + 4 * (lane & 3));
}
__device__ __forceinline__ void resid32_staged(const ConvArgs& a, long long vox0, int c0, const uint32_t* acc,
                                               const float* bias, float* stg, int lane, float4 (&s)[4]) {
#pragma unroll
    for (int q = 0; q < 4; ++q)
        *reinterpret_cast<float4*>(stg + lane * 16 + 4 * (q ^ ((lane >> 1) & 3))) =
            make_float4(__uint_as_float(acc[4 * q]) + bias[4 * q], __uint_as_float(acc[4 * q + 1]) + bias[4 * q + 1],
                        __uint_as_float(acc[4 * q + 2]) + bias[4 * q + 2],
                        __uint_as_float(acc[4 * q + 3]) + bias[4 * q + 3]);
    __syncwarp();
    const int c = lane & 3;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int v = (lane >> 2) + 8 * i;
        const float4 d = *reinterpret_cast<const float4*>(stg + v * 16 + 4 * (c ^ ((v >> 1) & 3)));
        s[i].x += d.x, s[i].y += d.y, s[i].z += d.z, s[i].w += d.w;
        const long long o = (vox0 + v) * 32 + c0 + 4 * c;
        *reinterpret_cast<float4*>(reinterpret_cast<float*>(a.pre) + o) = s[i];
        uint2 ob;
        __nv_bfloat162 lo = __floats2bfloat162_rn(s[i].x, s[i].y), hi = __floats2bfloat162_rn(s[i].z, s[i].w);
        ob.x = *reinterpret_cast<uint32_t*>(&lo);
        ob.y = *reinterpret_cast<uint32_t*>(&hi);
        *reinterpret_cast<uint2*>(reinterpret_cast<__nv_bfloat16*>(a.out) + o) = ob;
    }
    __syncwarp();  // staging reads done before the next row overwrites it
}

// ----------------------------------------------- pipelined scatter kernel
namespace ring {
constexpr int ZT = 128;                    // voxels per output row tile (MMA M)
constexpr int RZ = 160;                    // z rows (64 bytes each) per x-row run: z0 + i at row 16 + i
constexpr int RUN = RZ * 64;               // bytes per run (a multiple of 1024)
constexpr int NS = 5;                      // ring slots (one input row each)
constexpr int SLOT = 3 * RUN;              // bytes per slot: runs for x-1, x, x+1
constexpr int WB = 9 * 12 * 4 * 128;       // staged weights: [dx][dz][n/8 (12)][ci/8][8 n][8 ci]
constexpr int NBLK = 16;                   // accumulator blocks of 32 columns (a ring over output rows)
constexpr int NEPI = 8;                    // epilogue warps of a group
// groups of epilogue warps, which take alternate output rows: two for the GELU-backward
// epilogue, whose arithmetic and loads set the pace (8 x 256^3: 12.3 ms with one group, 8.2
// with two and its pre-activations loaded ahead). GELU is slower with two (8.3 -> 8.7).
__host__ __device__ constexpr int groups(int epi) { return epi == EVX_NN_EPI_GELU_BWD ? 2 : 1; }
__host__ __device__ constexpr int threads(int epi) { return (2 + NEPI * groups(epi)) * 32; }
constexpr int BAR = WB + NS * SLOT;        // barriers: full[NS], tfull[NBLK], tempty[NBLK]
constexpr int STG = (BAR + 8 * (NS + 2 * NBLK) + 16 + 15) & ~15;  // after the tensor-memory slot and abort flag
constexpr int STG_WARP = 32 * 16 * 4;      // per epilogue warp: [32 voxels][16 channels] FP32 staging
constexpr int SMEM = STG + NEPI * STG_WARP + 1024;  // + alignment
constexpr long long WAIT_BUDGET = 1LL << 31;
}  // namespace ring

struct RingArgs {
    ConvArgs a;
    int nzc;     // z chunks: ceil(Z / 128), the last of 64 voxels when Z is an odd multiple of 64
    int len;     // rows of a column: Y (columns (b, x, z chunk) walked along y) or X (columns (b, y, z chunk))
    int nseg;    // segments of a column
    int nunits;  // columns * nseg
};

// non-blocking probe of a phase (no suspend, unlike try_wait)
__device__ __forceinline__ bool mbar_test(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        " selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}

// bounded wait that also gives up once another role has aborted; a phase that has
// already completed is seen by the non-blocking probe first. mark: the flag's value
__device__ __forceinline__ bool ring_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag, int mark = 1) {
    if (mbar_test(bar, parity)) return true;
    const long long t0 = clock64();
    while (true) {
        if (mbar_try(bar, parity)) return true;
        if (*abort_flag) return false;
        if (clock64() - t0 > ring::WAIT_BUDGET) {
            *abort_flag = mark;
            atomicExch(&g_tc_timeout, 1);
            return false;
        }
    }
}

// as ring_wait for an event at the end of the kernel: gives up when another role has,
// or after 32 times the bound of a single pipeline wait
__device__ __forceinline__ bool ring_wait_long(uint32_t bar, uint32_t parity, volatile int* abort_flag) {
    const long long t0 = clock64();
    while (true) {
        if (mbar_try(bar, parity)) return true;
        if (*abort_flag) return false;
        if (clock64() - t0 > 32 * ring::WAIT_BUDGET) {
            *abort_flag = 1;
            atomicExch(&g_tc_timeout, 1);
            return false;
        }
    }
}

// unit u -> column bx = b * X + x (b * Y + y), z-chunk start z0, output rows ys .. ye-1
__device__ __forceinline__ void ring_unit(const RingArgs& r, int u, int& bx, int& z0, int& ys, int& ye) {
    const int seg = u % r.nseg, col = u / r.nseg;
    z0 = (col % r.nzc) * ring::ZT;
    bx = col / r.nzc;
    ys = (int)((long long)seg * r.len / r.nseg);
    ye = (int)((long long)(seg + 1) * r.len / r.nseg);
}

// accumulator block of virtual output row v: descending, so that the rows
// v + 2, v + 1, v fed by one input row are consecutive blocks
__device__ __forceinline__ uint32_t ring_blk(uint32_t v) { return (ring::NBLK - v % ring::NBLK) % ring::NBLK; }

// MMA q = 2 (3 dxi + dzi) + ks of an input row: descriptor offsets (16-byte
// units) of its A operand (from the slot's first run: z row 15 + dzi of run
// dxi, plus 32 bytes for the second K-step) and of its B operand (from the
// staged weights)
__host__ __device__ constexpr uint64_t ring_aoff(int q) {
    return (uint64_t)(((q >> 1) / 3) * (ring::RUN / 16) + (15 + (q >> 1) % 3) * 4 + 2 * (q & 1));
}
__host__ __device__ constexpr uint64_t ring_boff(int q) { return (uint64_t)(((q >> 1) * 12 * 4 + 2 * (q & 1)) * 8); }

__device__ __forceinline__ void tmem_st16_zero(uint32_t taddr) {
    const uint32_t z = 0;
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1};" ::"r"(taddr),
        "r"(z)
        : "memory");
}

// WX: columns are walked along x and may end in a 64-voxel chunk (a template parameter: as
// run-time values the two forms cost the Z % 128 = 0 convolutions 4 to 9%)
template <int EPI, bool WX>
__global__ void __launch_bounds__(ring::threads(EPI), 1)
    conv_ring_kernel(const __grid_constant__ CUtensorMap map, const __grid_constant__ CUtensorMap hmap, RingArgs r) {
    using namespace ring;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    unsigned char* sm = smem_raw + ((1024u - (smem_addr(smem_raw) & 1023u)) & 1023u);  // swizzle atoms: 1024-aligned
    unsigned char* swb = sm;
    unsigned char* sring = sm + WB;
    const uint32_t full = smem_addr(sm + BAR), tfull = full + 8 * NS, tempty = tfull + 8 * NBLK;
    uint32_t* tslot = reinterpret_cast<uint32_t*>(sm + BAR + 8 * (NS + 2 * NBLK));
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tslot + 1);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const ConvArgs& a = r.a;
    const int X = a.X, Y = a.Y, Z = a.Z;

    // weights [t][co][ci] -> [dx][dz][n = 32 (dy+1) + co][ci]: one input row feeds the output rows
    // y' + 1 (dy = -1), y' (dy = 0), y' - 1 (dy = +1) through N = 96 stacked columns (walking x:
    // x and y change places)
    for (int e = threadIdx.x; e < 9 * 96 * 4; e += threads(EPI)) {
        const int kg = e & 3, n = (e >> 2) % 96, dd = e / (96 * 4), dxi = dd / 3, dzi = dd % 3;
        const int t = WX ? 9 * (n >> 5) + 3 * dxi + dzi : 9 * dxi + 3 * (n >> 5) + dzi, co = n & 31;
        const uint4 v = *reinterpret_cast<const uint4*>(a.w + (t * 32 + co) * 32 + kg * 8);
        *reinterpret_cast<uint4*>(swb + (((dd * 12 + (n >> 3)) * 4 + kg) * 8 + (n & 7)) * 16) = v;
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(tslot)),
                     "n"(NBLK * 32)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (threadIdx.x == 0) {
        for (int s = 0; s < NS; ++s) mbar_init(full + 8 * s, 1);
        for (int c = 0; c < NBLK; ++c) {
            mbar_init(tfull + 8 * c, 1);
            mbar_init(tempty + 8 * c, NEPI);
        }
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // staged weights -> MMA operand reads
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tmem = *tslot;
    if (warp >= 2 && warp < 2 + NEPI) {  // every accumulator block starts at zero; the MMAs only accumulate
        const uint32_t tq = tmem + ((uint32_t)((warp & 3) * 32) << 16) + ((warp - 2) >> 2) * 16;
        for (int c = 0; c < NBLK; ++c) tmem_st16_zero(tq + c * 32);
        asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
    }
    fence_before();
    __syncthreads();
    fence_after();

    if (warp == 0) {
        // ---------------------------------------------------------- producer
        // A slot is refilled once the MMAs of the row it last held have completed:
        // the MMA warp's commit on that row's accumulator block (virtual row
        // vslot[slot]) already signals it, so the slot needs no barrier of its own.
        uint32_t k = 0, V = 0;  // slots issued; first virtual row of the unit
        uint32_t vslot[NS];
        bool ok = true;
        for (int u = blockIdx.x; u < r.nunits && ok; u += gridDim.x) {
            int bx, z0, ys, ye;
            ring_unit(r, u, bx, z0, ys, ye);
            const int across = WX ? Y : X, b = bx / across, x = bx - b * across;
            const int nz = WX ? min(ZT, Z - z0) : ZT;  // 128, or 64 in a last half chunk (its rows 64 .. are not loaded)
            for (int j = -1; j <= ye - ys; ++j) {
                const int yp = (ys + j + r.len) % r.len;
                const uint32_t slot = k % NS;
                uint32_t w_ok = 1;
                if (lane == 0 && k >= NS)
                    w_ok = ring_wait(tfull + 8 * ring_blk(vslot[slot]), (vslot[slot] / NBLK) & 1, abort_flag);
                vslot[slot] = V + (uint32_t)(j + 1);
                if (!__shfl_sync(0xffffffffu, w_ok, 0)) {
                    ok = false;
                    break;
                }
                if (lane == 0) {
                    const uint32_t base = smem_addr(sring + slot * SLOT);
                    const int zl = (z0 - 16 + Z) % Z, zr = (z0 + nz) % Z;  // periodic z halo: 16-row boxes
                    mbar_expect_tx(full + 8 * slot, 3 * (nz + 32) * 64);
#pragma unroll
                    for (int dxi = 0; dxi < 3; ++dxi) {
                        const int side = (x + dxi - 1 + across) % across;
                        const int cy = WX ? side : yp, cx = b * X + (WX ? yp : side);
                        const uint32_t run = base + dxi * RUN;
                        tma_load4(run + 16 * 64, &map, 0, z0, cy, cx, full + 8 * slot);
                        if (WX && nz == ZT) tma_load4(run + (16 + 64) * 64, &map, 0, z0 + 64, cy, cx, full + 8 * slot);
                        tma_load4(run, &hmap, 0, zl, cy, cx, full + 8 * slot);
                        tma_load4(run + (16 + nz) * 64, &hmap, 0, zr, cy, cx, full + 8 * slot);
                    }
                }
                __syncwarp();
                ++k;
            }
            V += (uint32_t)(ye - ys) + 4;
        }
        if (!ok && lane == 0)  // let this CTA's copies in flight land before it exits (bounded)
            for (uint32_t q = (k > (uint32_t)NS ? k - NS : 0); q < k; ++q) tc_wait(full + 8 * (q % NS), (q / NS) & 1);
    } else if (warp == 1) {
        // ------------------------------------------------------- MMA issuer
        // The whole warp walks the schedule (descriptors stay warp-uniform);
        // lane 0 waits, issues and commits. Input row i of a unit (y' = ys-1+i)
        // feeds virtual rows V+i+2, V+i+1, V+i (output rows y'+1, y', y'-1);
        // virtual rows V .. V+L+3 hold output rows ys-2 .. ye+1, of which the
        // first and last two are partial and discarded.
        constexpr uint32_t I96 = idesc_bf16(ZT, 96), I64 = idesc_bf16(ZT, 64), I32 = idesc_bf16(ZT, 32);
        const uint32_t ring0 = smem_addr(sring);
        const uint64_t bdesc0 = sdesc(smem_addr(swb), 128, 512);
        uint32_t k = 0, V = 0, last_v = 0;
        uint32_t vready = NBLK - 1;  // virtual rows <= vready have a free (zeroed) accumulator block
        bool ok = true, issued = false;
        for (int u = blockIdx.x; u < r.nunits && ok; u += gridDim.x) {
            int bx, z0, ys, ye;
            ring_unit(r, u, bx, z0, ys, ye);
            const uint32_t L = (uint32_t)(ye - ys);
            for (uint32_t i = 0; i <= L + 1; ++i, ++k) {
                // blocks are claimed 8 rows at a time (rows up to V+i+9, freed by the epilogue
                // once it has read rows up to V+i-7), so the tensor-memory fence that orders
                // the epilogue's reads before these MMAs runs once per 8 input rows. Every
                // epilogue warp frees its rows in order, so the phase of the last claimed block
                // (row V+i-7 freed by all warps of its group) implies the group's earlier ones:
                // one probe per group, not 8, of a barrier the tensor core's operand reads make
                // slow to reach.
                const bool claim = V + i + 2 > vready;
                uint32_t w_ok = 1;
                if (lane == 0) {
                    const uint32_t vc = V + i + 9;
                    if (claim) w_ok = ring_wait(tempty + 8 * ring_blk(vc), ((vc / NBLK) & 1) ^ 1, abort_flag);
                    if (groups(EPI) == 2 && claim && w_ok)  // the other group's last claimed row
                        w_ok = ring_wait(tempty + 8 * ring_blk(vc - 1), (((vc - 1) / NBLK) & 1) ^ 1, abort_flag);
                    if (w_ok) w_ok = ring_wait(full + 8 * (k % NS), (k / NS) & 1, abort_flag);
                }
                if (!__shfl_sync(0xffffffffu, w_ok, 0)) {
                    ok = false;
                    break;
                }
                if (claim) {
                    vready = V + i + 9;
                    fence_after();
                }
                const uint64_t adesc = sdesc_sw64(ring0 + (k % NS) * SLOT);
                const uint32_t b0 = ring_blk(V + i + 2);  // blocks b0, b0+1, b0+2 (mod 16)
                // 18 MMAs (dx, dz, ks); where the three blocks wrap past the last
                // column, each splits into two. One (warp-uniform) branch per input
                // row keeps the unrolled issue sequences free of per-MMA control
                // flow; the warp stays converged and lane 0 issues (and commits).
                {
                    if (b0 <= NBLK - 3) {
#pragma unroll
                        for (int q = 0; q < 18; ++q)
                            tc_mma_lane0(tmem + b0 * 32, adesc + ring_aoff(q), bdesc0 + ring_boff(q), I96);
                    } else if (b0 == NBLK - 2) {
#pragma unroll
                        for (int q = 0; q < 18; ++q) {
                            tc_mma_lane0(tmem + b0 * 32, adesc + ring_aoff(q), bdesc0 + ring_boff(q), I64);
                            tc_mma_lane0(tmem, adesc + ring_aoff(q), bdesc0 + ring_boff(q) + 8 * 4 * 8, I32);
                        }
                    } else {
#pragma unroll
                        for (int q = 0; q < 18; ++q) {
                            tc_mma_lane0(tmem + b0 * 32, adesc + ring_aoff(q), bdesc0 + ring_boff(q), I32);
                            tc_mma_lane0(tmem, adesc + ring_aoff(q), bdesc0 + ring_boff(q) + 4 * 4 * 8, I64);
                        }
                    }
                }
                if (lane == 0) {
                    tc_commit(tfull + 8 * ring_blk(V + i));  // virtual row V+i has all its inputs; slot k is free
                    if (i == L + 1) {
                        tc_commit(tfull + 8 * ring_blk(V + L + 2));
                        tc_commit(tfull + 8 * ring_blk(V + L + 3));
                    }
                }
                issued = true;
                last_v = V + i;
                __syncwarp();
            }
            V += L + 4;
        }
        if (!ok && lane == 0 && issued)  // let the last MMAs land before the accumulators are freed (bounded)
            tc_wait(tfull + 8 * ring_blk(last_v), (last_v / NBLK) & 1);
        __syncwarp();
    } else {
        // --------------------------------------------------------- epilogue
        // Virtual row v belongs to group v mod G. The FP32 stream and the pre-activations of
        // GELU' are loaded one row of the group ahead (RESID32 9.9 -> 9.25 ms at 8 x 256^3; the
        // BF16 residuals of RESID gain nothing: 6.6 -> 7.2).
        constexpr int G = groups(EPI);
        constexpr bool STREAM = EPI == EVX_NN_EPI_RESID32, AHEAD = EPI == EVX_NN_EPI_GELU_BWD;
        const int q4 = warp & 3, h = ((warp - 2) & 7) >> 2;  // accumulator lanes 32 q4 .., columns 16 h ..
        const uint32_t grp = G == 2 ? (warp - 2) >> 3 : 0;
        float* stg = reinterpret_cast<float*>(sm + STG + (warp - 2) * STG_WARP);
        float bias[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) bias[i] = a.bias ? a.bias[h * 16 + i] : 0.f;
        uint32_t V = 0;
        bool ok = true;
        for (int u = blockIdx.x; u < r.nunits && ok; u += gridDim.x) {
            int bx, z0, ys, ye;
            ring_unit(r, u, bx, z0, ys, ye);
            const int L = ye - ys;
            // voxel of the row's lane 0 and the distance to the next row's
            const long long row0 = WX ? ((long long)(bx / Y) * X + ys) * Y + bx % Y : (long long)bx * Y + ys;
            const long long step = WX ? (long long)Y * Z : Z;
            const int j0 = G == 2 ? (int)((grp - V) & 1) : 0;
            long long vox0 = row0 * Z + z0 + q4 * 32 + (j0 - 2) * step;  // of virtual row jv
            // rows that are stored; a half chunk's lanes 64 .. are not voxels
            auto stored = [&](int j) { return j >= 2 && j < L + 2 && (!WX || z0 + q4 * 32 < Z); };
            uint4 pf[2], pfn[2];
            float4 sf[4], sfn[4];
            for (int jv = j0; jv < L + 4; jv += G, vox0 += G * step) {
                const uint32_t v = V + jv, blk = ring_blk(v);
                if (AHEAD || STREAM) {  // (the first stored row of a group is never its first row)
#pragma unroll
                    for (int i = 0; i < 2; ++i) pf[i] = pfn[i];
#pragma unroll
                    for (int i = 0; i < 4; ++i) sf[i] = sfn[i];
                    if (stored(jv + G)) {
                        const long long vn = vox0 + G * step;
                        if (STREAM) resid32_load(a, vn, h * 16, lane, sfn);
                        if (AHEAD)
#pragma unroll
                            for (int i = 0; i < 2; ++i)
                                pfn[i] = *reinterpret_cast<const uint4*>(a.pre + (vn + lane) * 32 + h * 16 + 8 * i);
                    }
                }
                uint32_t w_ok = 1;
                if (lane == 0) w_ok = ring_wait(tfull + 8 * blk, (v / NBLK) & 1, abort_flag);
                if (!__shfl_sync(0xffffffffu, w_ok, 0)) {
                    ok = false;
                    break;
                }
                fence_after();
                uint32_t acc[16];
                const uint32_t tq = tmem + ((uint32_t)(q4 * 32) << 16) + blk * 32 + h * 16;
                tmem_ld16(tq, acc);
                asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                tmem_st16_zero(tq);
                asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
                fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(tempty + 8 * blk);
                if (stored(jv)) {
                    if constexpr (STREAM)
                        resid32_staged(a, vox0, h * 16, acc, bias, stg, lane, sf);
                    else
                        epilogue_store<EPI, 16>(a, vox0 + lane, h * 16, acc, bias, pf);
                }
            }
            V += (uint32_t)L + 4;
        }
    }
    fence_before();
    __syncthreads();
    fence_after();
    if (warp == 1)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "n"(NBLK * 32) : "memory");
}

// ------------------------------------------------------- weight gradient
// dW[t][co][ci] = sum_v dY(v, co) X(v + off_t, ci): a GEMM whose K is the voxels.
// Both operands lie in shared memory as TMA writes them, rows of one voxel's 32
// channels (64 bytes, 64-byte swizzle), so the MMA reads both with the channels
// contiguous (MN-major) and no transposition. One input row (x' = x - 1 .. x + 1,
// y', 128 z) meets the three output rows y' - 1, y', y' + 1:
//   A (M = 128): four groups of 32 ci, one z row (64 bytes) apart: dz = -1, 0, +1
//                and a fourth that is not used
//   B (N = 96):  three groups of 32 co, one dY row slot apart: dy = +1, 0, -1
//   K = 16 voxels per MMA: 3 dx x 8 = 24 MMAs per row into 96 columns of tensor
//   memory per dx (acc_col), accumulated over the CTA's rows (27 taps at once)
// An input row costs about what a convolution's does (18 MMAs of N = 96); a unit's
// rows each count in full (the halo is on the dY rows: 8 of the 38 KB a row
// loads). The mma.sync kernel it replaces for 32 -> 32 re-read its fragments from
// shared memory for every tap: 382 us at 64 x 96 x 128 and 3.71 ms at 4 x 128^3 with the
// sum of the partials, this kernel 78 us and 0.61 ms (error against 64 bits 5.63e-6 ->
// 3.96e-6 at 64 x 96 x 128).
//   warp 0 producer, warp 1 MMA issuer, warps 2..5 write the CTA's partial sums.
namespace wg {
constexpr int NS = 4;                        // input-row slots (3 runs each, as in the ring)
constexpr int NR = 11;                       // dY row slots (128 z x 64 bytes)
constexpr int DYROW = 128 * 64;
constexpr int XOFF = NR * DYROW;
constexpr int BAR = XOFF + NS * ring::SLOT;  // full[NS], free[NS], done
constexpr int SMEM = BAR + 8 * (2 * NS + 1) + 16 + 1024;
constexpr int NTH = 6 * 32;
constexpr uint32_t COLS = 512;
// column of dx's accumulator for the CTA's input row k: dx = -1 and 0 have one for even and
// one for odd rows (5 x 96 of the 512 columns). The tensor core truncates as it adds, so the
// error grows with the length of a chain: with one accumulator each, dW was up to 1.8%
// further from 64 bits than the mma.sync kernel's.
__device__ __forceinline__ uint32_t acc_col(int dx, uint32_t k) { return dx * 96 + (dx < 2 && (k & 1) ? 288 : 0); }
}  // namespace wg

struct WgArgs {
    float* partials;  // [grid][27][32][32]
    int B, X, Y, Z, nzc, zbox, nseg, nunits;
};

// MN-major operand in the 64-byte swizzle layout: 8 K rows of 64 bytes per 512-byte
// group (stride byte offset), groups of 32 channels mn_stride bytes apart (leading)
__device__ __forceinline__ uint64_t sdesc_mn64(uint32_t saddr, uint32_t mn_stride) {
    return sdesc(saddr, mn_stride, 512) | (4ull << 61);
}
__host__ __device__ constexpr uint32_t idesc_bf16_mn(int M, int N) { return idesc_bf16(M, N) | (1u << 15) | (1u << 16); }

__device__ __forceinline__ void tc_mma_lane0_acc(uint32_t dtmem, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
    asm volatile(
        "{\n .reg .pred p, q;\n .reg .u32 l;\n mov.u32 l, %%laneid;\n setp.eq.u32 p, l, 0;\n"
        " setp.ne.b32 q, %4, 0;\n @p tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, q;\n}\n" ::"r"(dtmem),
        "l"(a), "l"(b), "r"(idesc), "r"(acc)
        : "memory");
}

__device__ __forceinline__ void wg_unit(const WgArgs& r, int u, int& bx, int& z0, int& ys, int& ye) {
    const int seg = u % r.nseg, col = u / r.nseg;
    z0 = (col % r.nzc) * ring::ZT;
    bx = col / r.nzc;
    ys = (int)((long long)seg * r.Y / r.nseg);
    ye = (int)((long long)(seg + 1) * r.Y / r.nseg);
}

__global__ void __launch_bounds__(wg::NTH, 1)
    conv_wgrad_tc_kernel(const __grid_constant__ CUtensorMap xmap, const __grid_constant__ CUtensorMap xhalo,
                         const __grid_constant__ CUtensorMap dymap, WgArgs r) {
    using namespace wg;
    using ring::RUN;
    using ring::SLOT;
    using ring::ZT;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    unsigned char* sm = smem_raw + ((1024u - (smem_addr(smem_raw) & 1023u)) & 1023u);
    const uint32_t sdy = smem_addr(sm), sx = smem_addr(sm + XOFF);
    const uint32_t full = smem_addr(sm + BAR), freeb = full + 8 * NS, done = freeb + 8 * NS;
    uint32_t* tslot = reinterpret_cast<uint32_t*>(sm + BAR + 8 * (2 * NS + 1));
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tslot + 1);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int X = r.X, Y = r.Y, Z = r.Z;
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(tslot)), "n"(COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (threadIdx.x == 0) {
        for (int s = 0; s < 2 * NS + 1; ++s) mbar_init(full + 8 * s, 1);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tmem = *tslot;
    if (warp == 0) {
        // ---------------------------------------------------------- producer
        // Input row k takes slot k % NS once row k - NS has been consumed; dY row q takes
        // slot q % NR once the last input row that reads q - NR has been.
        uint32_t k = 0, q = 0;
        uint32_t last[NR];  // input row (plus one) that last reads the dY row held by a slot
#pragma unroll
        for (int i = 0; i < NR; ++i) last[i] = 0;
        if (lane == 0) {
            uint32_t seen = 0;  // input rows known to be consumed
            bool ok = true;
            auto consumed = [&](uint32_t n) {  // wait until the first n input rows are
                if (n <= seen) return true;
                if (!ring_wait(freeb + 8 * ((n - 1) % NS), ((n - 1) / NS) & 1, abort_flag)) return false;
                seen = n;
                return true;
            };
            for (int u = blockIdx.x; u < r.nunits && ok; u += gridDim.x) {
                int bx, z0, ys, ye;
                wg_unit(r, u, bx, z0, ys, ye);
                const int b = bx / X, x = bx - b * X, L = ye - ys;
                const int nz = min(ZT, Z - z0);
                const int zl = (z0 - 16 + Z) % Z, zr = (z0 + nz) % Z;
                for (int i = 0; i < L; ++i, ++k) {
                    if (k >= (uint32_t)NS && !(ok = consumed(k - NS + 1))) break;
                    const int nd = i == 0 ? 3 : 1;  // dY rows that arrive with this input row
                    for (int d = 0; d < nd && ok; ++d) ok = consumed(last[(q + d) % NR]);
                    if (!ok) break;
                    const uint32_t bar = full + 8 * (k % NS);
                    mbar_expect_tx(bar, 3 * (nz + 32) * 64 + nd * nz * 64);
                    for (int d = 0; d < nd; ++d, ++q) {
                        const int j = i == 0 ? d : i + 2;  // dY row ys - 1 + j, read by input rows j - 2 .. j of the unit
                        const int yd = (ys - 1 + j + Y) % Y;
                        const uint32_t dst = sdy + (q % NR) * DYROW;
                        last[q % NR] = k - i + min(j, L - 1) + 1;
                        tma_load4(dst, &dymap, 0, z0, yd, bx, bar);
                        if (nz > r.zbox) tma_load4(dst + 64 * 64, &dymap, 0, z0 + 64, yd, bx, bar);
                    }
                    const int yp = ys + i;
                    const uint32_t base = sx + (k % NS) * SLOT;
#pragma unroll
                    for (int dxi = 0; dxi < 3; ++dxi) {
                        const int cx = b * X + (x + dxi - 1 + X) % X;
                        const uint32_t run = base + dxi * RUN;
                        tma_load4(run + 16 * 64, &xmap, 0, z0, yp, cx, bar);
                        if (nz > r.zbox) tma_load4(run + (16 + 64) * 64, &xmap, 0, z0 + 64, yp, cx, bar);
                        tma_load4(run, &xhalo, 0, zl, yp, cx, bar);
                        tma_load4(run + (16 + nz) * 64, &xhalo, 0, zr, yp, cx, bar);
                    }
                }
            }
            if (!ok)  // let the copies in flight land before the CTA exits (bounded)
                for (uint32_t m = (k > (uint32_t)NS ? k - NS : 0); m < k; ++m) tc_wait(full + 8 * (m % NS), (m / NS) & 1);
        }
        __syncwarp();
    } else if (warp == 1) {
        // ------------------------------------------------------- MMA issuer
        constexpr uint32_t I96 = idesc_bf16_mn(128, 96), I64 = idesc_bf16_mn(128, 64), I32 = idesc_bf16_mn(128, 32);
        uint32_t k = 0, q = 0;
        bool ok = true;
        for (int u = blockIdx.x; u < r.nunits && ok; u += gridDim.x) {
            int bx, z0, ys, ye;
            wg_unit(r, u, bx, z0, ys, ye);
            const int L = ye - ys, ksteps = min(ZT, Z - z0) / 16;
            for (int i = 0; i < L; ++i, ++k, ++q) {
                uint32_t w_ok = 1;
                if (lane == 0) w_ok = ring_wait(full + 8 * (k % NS), (k / NS) & 1, abort_flag);
                if (!__shfl_sync(0xffffffffu, w_ok, 0)) {
                    ok = false;
                    break;
                }
                const uint32_t s0 = q % NR;  // slots of the dY rows y' - 1, y', y' + 1: s0, s0 + 1, s0 + 2 (mod NR)
                const uint64_t a0 = sdesc_mn64(sx + (k % NS) * SLOT + 15 * 64, 64);
                const uint64_t b0 = sdesc_mn64(sdy + s0 * DYROW, DYROW), bw = sdesc_mn64(sdy, DYROW);
                if (s0 <= NR - 3) {
                    for (int ks = 0; ks < ksteps; ++ks)
#pragma unroll
                        for (int dx = 0; dx < 3; ++dx)
                            tc_mma_lane0_acc(tmem + acc_col(dx, k), a0 + (dx * RUN + ks * 1024) / 16, b0 + ks * 64, I96,
                                             k > (dx < 2) || ks > 0);
                } else {  // the three slots wrap (never at k = 0 or 1): N = 64 + 32 or 32 + 64
                    const uint32_t n1 = (NR - s0) * 32, i1 = n1 == 64 ? I64 : I32, i2 = n1 == 64 ? I32 : I64;
                    for (int ks = 0; ks < ksteps; ++ks)
#pragma unroll
                        for (int dx = 0; dx < 3; ++dx) {
                            const uint64_t ad = a0 + (dx * RUN + ks * 1024) / 16;
                            tc_mma_lane0_acc(tmem + acc_col(dx, k), ad, b0 + ks * 64, i1, 1);
                            tc_mma_lane0_acc(tmem + acc_col(dx, k) + n1, ad, bw + ks * 64, i2, 1);
                        }
                }
                if (lane == 0) tc_commit(freeb + 8 * (k % NS));
                __syncwarp();
            }
            q += 2;  // the unit loaded L + 2 dY rows
        }
        if (lane == 0) {
            tc_commit(done);  // every MMA issued has completed
            if (!ok) tc_wait(done, 0);
        }
        __syncwarp();
    } else {
        // --------------------------------------------------- partial sums
        const int dzi = warp & 3;  // accumulator lanes 32 dzi .. : (dz, ci = lane); the fourth group is not used
        uint32_t w_ok = 1;
        if (lane == 0) w_ok = ring_wait_long(done, 0, abort_flag);
        w_ok = __shfl_sync(0xffffffffu, w_ok, 0);
        fence_after();
        if (w_ok && dzi < 3) {
            float* P = r.partials + (long long)blockIdx.x * 27 * 32 * 32;
            int rows = 0;  // the odd rows' accumulators hold sums if there is a second row
            for (int u = blockIdx.x; u < r.nunits && rows < 2; u += gridDim.x) {
                int bx, z0, ys, ye;
                wg_unit(r, u, bx, z0, ys, ye);
                rows += ye - ys;
            }
#pragma unroll 1
            for (int g = 0; g < 18; ++g) {  // 16 output channels of one (dx, dy)
                const int dxi = g / 6, j = (g / 2) % 3, co = (g & 1) * 16;
                uint32_t acc[16];
                const uint32_t at = tmem + ((uint32_t)(dzi * 32) << 16) + j * 32 + co;
                tmem_ld16(at + acc_col(dxi, 0), acc);
                asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                if (dxi < 2 && rows > 1) {
                    uint32_t odd[16];
                    tmem_ld16(at + acc_col(dxi, 1), odd);
                    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
                    for (int c = 0; c < 16; ++c)
                        acc[c] = __float_as_uint(__uint_as_float(acc[c]) + __uint_as_float(odd[c]));
                }
                const int t = 9 * dxi + 3 * (2 - j) + dzi;
#pragma unroll
                for (int c = 0; c < 16; ++c) P[(t * 32 + co + c) * 32 + lane] = __uint_as_float(acc[c]);
            }
        }
    }
    fence_before();
    __syncthreads();
    fence_after();
    if (warp == 1)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "n"(COLS) : "memory");
}

// --------------------------------------------------------------- projection
// out(v) = bias(0) + sum_t sum_ci w[t][0][ci] h32(v + off_t, ci), FP32 stream: a
// CTA owns 16 rows (y) x 32 z and walks x. Lane = channel; a warp owns two rows.
// Each input plane is read once (TMA, two buffers) and each of its values once
// from shared memory, for the three output planes it feeds: their 3 x 2 x 32
// partial sums stay in registers and move on by one plane per step. A lane adds
// its taps in the order (dx, dy, dz), then the lanes are summed by a butterfly.
// Bound by the 864 FMAs per voxel (2.9 ms at 8 x 256^3); the plane halo is 1.2 x.
// One warp per 2 x 32 outputs without the walk read every value three times from
// shared memory or L1 and six times from L2: 10.6 ms at 8 x 256^3, 6.3 now.
namespace pj {
constexpr int ROWS = 16, ZT = 32, NT = 256;
constexpr int PROW = (ZT + 2) * 32;            // floats per plane row: z0 - 1 .. z0 + 32, 32 channels
constexpr int PLANE = (ROWS + 2) * PROW * 4;   // bytes
constexpr int BAR = 2 * PLANE;
constexpr int SMEM = BAR + 2 * 8 + 16;
}  // namespace pj

struct PjArgs {
    const __nv_bfloat16* w;
    int wcout;
    const float* bias;
    float* out;
    int B, X, Y, Z, nyt, nseg, nunits;
};

__device__ __forceinline__ float pj_lane_sums(float (&v)[32], int lane) {  // lane l: the lanes' sum of v[l]
#pragma unroll
    for (int off = 16; off >= 1; off >>= 1) {
        const bool upper = lane & off;
#pragma unroll
        for (int k = 0; k < off; ++k) {
            const float send = upper ? v[k] : v[k + off];
            const float keep = upper ? v[k + off] : v[k];
            v[k] = keep + __shfl_xor_sync(0xffffffffu, send, off);
        }
    }
    return v[0];
}

__global__ void __launch_bounds__(pj::NT, 1)
    project_walk_kernel(const __grid_constant__ CUtensorMap map, const __grid_constant__ CUtensorMap hmap, PjArgs r) {
    using namespace pj;
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    __shared__ float ws[27][32];  // w[t][0][ci]
    const uint32_t full = smem_addr(smem_raw + BAR);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(smem_raw + BAR + 16);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int X = r.X, Y = r.Y, Z = r.Z;
    for (int i = threadIdx.x; i < 27 * 32; i += NT)
        ws[i >> 5][i & 31] = __bfloat162float(r.w[(long long)(i >> 5) * r.wcout * 32 + (i & 31)]);
    if (threadIdx.x == 0) {
        mbar_init(full, 1);
        mbar_init(full + 8, 1);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    const float b0 = r.bias ? r.bias[0] : 0.f;
    __syncthreads();
    uint32_t k = 0;  // planes consumed
    bool go = true;
    for (int u = blockIdx.x; u < r.nunits && go; u += gridDim.x) {
        const int seg = u % r.nseg;
        int c = u / r.nseg;
        const int z0 = (c % (Z / ZT)) * ZT;
        c /= Z / ZT;
        const int y0 = (c % r.nyt) * ROWS, b = c / r.nyt;
        const int xs = (int)((long long)seg * X / r.nseg), xe = (int)((long long)(seg + 1) * X / r.nseg);
        const int np = xe - xs + 2;  // input planes xs - 1 .. xe
        // plane q of the unit into buffer kq & 1: warp w the rows w, w + 8, w + 16 (a lane each)
        auto load = [&](int q, uint32_t kq) {
            const uint32_t bar = full + 8 * (kq & 1);
            const int yr = warp + 8 * lane;
            if (threadIdx.x == 0) mbar_expect_tx(bar, PLANE);
            if (lane < 3 && yr < ROWS + 2) {
                const int bx = b * X + (xs - 1 + q + X) % X, y = (y0 + yr - 1 + Y) % Y;
                const uint32_t row = smem_addr(smem_raw) + (kq & 1) * PLANE + yr * PROW * 4;
                tma_load4(row + 128, &map, 0, z0, y, bx, bar);
                tma_load4(row, &hmap, 0, (z0 - 1 + Z) % Z, y, bx, bar);
                tma_load4(row + (ZT + 1) * 128, &hmap, 0, (z0 + ZT) % Z, y, bx, bar);
            }
            __syncwarp();
        };
        load(0, k);
        load(1, k + 1);
        float acc[3][2][32];  // output planes p - 1, p, p + 1 of input plane p
#pragma unroll
        for (int d = 0; d < 3; ++d)
#pragma unroll
            for (int j = 0; j < 32; ++j) acc[d][0][j] = acc[d][1][j] = 0.f;
        for (int q = 0; q < np; ++q, ++k) {
            (void)ring_wait(full + 8 * (k & 1), (k >> 1) & 1, abort_flag, (int)k + 1);  // seen in the flag below
            const float* pl = reinterpret_cast<const float*>(smem_raw + (k & 1) * PLANE) + (2 * warp) * PROW + lane;
#pragma unroll
            for (int yy = 0; yy < 4; ++yy) {
                float hv[ZT + 2];
#pragma unroll
                for (int j = 0; j < ZT + 2; ++j) hv[j] = pl[yy * PROW + j * 32];
#pragma unroll
                for (int o = 0; o < 2; ++o) {
                    const int dy = yy - o;
                    if (dy < 0 || dy > 2) continue;
#pragma unroll
                    for (int d = 0; d < 3; ++d)  // output plane p - 1 + d takes this plane as its dx = 1 - d
#pragma unroll
                        for (int dz = 0; dz < 3; ++dz) {
                            const float wt = ws[9 * (2 - d) + 3 * dy + dz][lane];
#pragma unroll
                            for (int j = 0; j < 32; ++j) acc[d][o][j] = fmaf(wt, hv[j + dz], acc[d][o][j]);
                        }
                }
            }
            __syncthreads();  // the plane has been read
            // a wait that ran out in any thread: nothing is loaded or stored from here on. Every thread
            // finds the same: a plane's mark is set before its barrier or not at all
            const uint32_t mark = *abort_flag;
            go = mark == 0 || mark > k + 1;
            if (go && q + 2 < np) load(q + 2, k + 2);
            if (go && q >= 2) {
                const int x = xs + q - 2, y = y0 + 2 * warp;
#pragma unroll
                for (int o = 0; o < 2; ++o) {
                    const float sum = pj_lane_sums(acc[0][o], lane);
                    if (y + o < Y) r.out[(((long long)b * X + x) * Y + y + o) * Z + z0 + lane] = sum + b0;
                }
            }
#pragma unroll
            for (int o = 0; o < 2; ++o)
#pragma unroll
                for (int j = 0; j < 32; ++j) {
                    acc[0][o][j] = acc[1][o][j];
                    acc[1][o][j] = acc[2][o][j];
                    acc[2][o][j] = 0.f;
                }
        }
    }
    if (!go && threadIdx.x == 0)  // the copies in flight, of the late plane and the next of its unit, land first (bounded)
        for (uint32_t m = (uint32_t)*abort_flag - 1, end = min(m + 2, k); m < end; ++m) tc_wait(full + 8 * (m & 1), (m >> 1) & 1);
}

}  // namespace evxnn

// =================================================================== host
namespace {
using namespace evxnn;

PFN_cuTensorMapEncodeTiled_v12000 nn_encode_fn() {
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    static bool tried = false;
    if (!tried) {
        tried = true;
        void* ptr = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &ptr, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = (PFN_cuTensorMapEncodeTiled_v12000)ptr;
        else
            cudaGetLastError();
    }
    return fn;
}

// activations [B X][Y][Z][32] as a 4D BF16 tensor (32 channels, Z, Y, B X), box 32 channels x zrows z,
// written to shared memory in the 64-byte swizzle layout
bool act_map(CUtensorMap* m, const __nv_bfloat16* act, int B, int X, int Y, int Z, int zrows) {
    auto fn = nn_encode_fn();
    if (!fn || ((uintptr_t)act & 15)) return false;
    const cuuint64_t dims[4] = {32, (cuuint64_t)Z, (cuuint64_t)Y, (cuuint64_t)B * X};
    const cuuint64_t strides[3] = {64, (cuuint64_t)Z * 64, (cuuint64_t)Y * Z * 64};
    const cuuint32_t box[4] = {32, (cuuint32_t)zrows, 1, 1};
    const cuuint32_t estr[4] = {1, 1, 1, 1};
    return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<__nv_bfloat16*>(act), dims, strides, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// FP32 stream [B X][Y][Z][32] as a 4D tensor, box 32 channels x zrows z
bool stream_map(CUtensorMap* m, const float* h32, int B, int X, int Y, int Z, int zrows) {
    auto fn = nn_encode_fn();
    if (!fn || ((uintptr_t)h32 & 15)) return false;
    const cuuint64_t dims[4] = {32, (cuuint64_t)Z, (cuuint64_t)Y, (cuuint64_t)B * X};
    const cuuint64_t strides[3] = {128, (cuuint64_t)Z * 128, (cuuint64_t)Y * Z * 128};
    const cuuint32_t box[4] = {32, (cuuint32_t)zrows, 1, 1};
    const cuuint32_t estr[4] = {1, 1, 1, 1};
    return fn(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, const_cast<float*>(h32), dims, strides, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// segments of at least min_rows rows that columns are split into: the split with the least
// work on the busiest CTA, a segment of n rows costing n + extra
int segments(long long ncol, int len, int ctas, int extra, int min_rows = 8) {
    int nseg = 1;
    long long best = 0;
    for (int s = 1; s == 1 || s <= len / min_rows; ++s) {
        const long long rows = (ncol * s + ctas - 1) / ctas * ((len + s - 1) / s + extra);
        if (s == 1 || rows < best) {
            best = rows;
            nseg = s;
        }
    }
    return nseg;
}

template <int EPI, bool WX>
cudaError_t launch_walk(const ConvArgs& a, cudaStream_t st, int sms) {
    RingArgs r{};
    r.a = a;
    r.nzc = (a.Z + ring::ZT - 1) / ring::ZT;
    CUtensorMap map, hmap;  // with a half chunk the main box has 64 rows
    if (!act_map(&map, a.in, a.B, a.X, a.Y, a.Z, WX ? 64 : ring::ZT) || !act_map(&hmap, a.in, a.B, a.X, a.Y, a.Z, 16))
        return cudaErrorInvalidValue;
    r.len = WX ? a.X : a.Y;
    const long long ncol = (long long)a.B * (WX ? a.Y : a.X) * r.nzc;
    const int nseg = segments(ncol, r.len, sms, 2, 2);
    if (ncol * nseg > (1LL << 30)) return cudaErrorInvalidValue;  // unit index would overflow int
    r.nseg = nseg;
    r.nunits = (int)(ncol * nseg);
    cudaError_t e =
        cudaFuncSetAttribute(conv_ring_kernel<EPI, WX>, cudaFuncAttributeMaxDynamicSharedMemorySize, ring::SMEM);
    if (e != cudaSuccess) return e;
    conv_ring_kernel<EPI, WX><<<std::min(r.nunits, sms), ring::threads(EPI), ring::SMEM, st>>>(map, hmap, r);
    return cudaGetLastError();
}

template <int EPI>
cudaError_t launch_ring(const ConvArgs& a, cudaStream_t st, int sms) {
    return a.Z % ring::ZT ? launch_walk<EPI, true>(a, st, sms) : launch_walk<EPI, false>(a, st, sms);
}
}  // namespace

namespace evxnn {

cudaError_t conv32_tc(const ConvArgs& a, int epilogue, cudaStream_t st, int sms) {
    switch (epilogue) {
        case EVX_NN_EPI_PLAIN: return launch_ring<EVX_NN_EPI_PLAIN>(a, st, sms);
        case EVX_NN_EPI_GELU: return launch_ring<EVX_NN_EPI_GELU>(a, st, sms);
        case EVX_NN_EPI_RESID: return launch_ring<EVX_NN_EPI_RESID>(a, st, sms);
        case EVX_NN_EPI_GELU_BWD: return launch_ring<EVX_NN_EPI_GELU_BWD>(a, st, sms);
        case EVX_NN_EPI_RESID32: return launch_ring<EVX_NN_EPI_RESID32>(a, st, sms);
    }
    return cudaErrorInvalidValue;
}

// (b, y tile, z tile) columns of the walking projection
static long long project32_columns(int B, int Y, int Z) { return (long long)B * ((Y + pj::ROWS - 1) / pj::ROWS) * (Z / pj::ZT); }

long long project32_planes(int B, int X, int Y, int Z, int sms) {
    const long long ncol = project32_columns(B, Y, Z);
    const int nseg = segments(ncol, X, sms, 2);
    return (ncol * nseg + sms - 1) / sms * ((X + nseg - 1) / nseg + 2);
}

cudaError_t project32_walk(const float* h32, const __nv_bfloat16* w, int wcout, const float* bias, float* out, int B, int X,
                           int Y, int Z, cudaStream_t st, int sms) {
    PjArgs r{};
    r.w = w, r.wcout = wcout, r.bias = bias, r.out = out;
    r.B = B, r.X = X, r.Y = Y, r.Z = Z;
    r.nyt = (Y + pj::ROWS - 1) / pj::ROWS;
    CUtensorMap m, hm;
    if (!stream_map(&m, h32, B, X, Y, Z, pj::ZT) || !stream_map(&hm, h32, B, X, Y, Z, 1)) return cudaErrorInvalidValue;
    const long long ncol = project32_columns(B, Y, Z);
    r.nseg = segments(ncol, X, sms, 2);
    if (ncol * r.nseg > (1LL << 30)) return cudaErrorInvalidValue;  // unit index would overflow int
    r.nunits = (int)(ncol * r.nseg);
    cudaError_t e = cudaFuncSetAttribute(project_walk_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, pj::SMEM);
    if (e != cudaSuccess) return e;
    project_walk_kernel<<<std::min(r.nunits, sms), pj::NT, pj::SMEM, st>>>(m, hm, r);
    return cudaGetLastError();
}

cudaError_t wgrad32_tc(const __nv_bfloat16* dy, const __nv_bfloat16* x, float* partials, int max_ctas, int B, int X, int Y,
                       int Z, cudaStream_t st, int sms, int* ctas) {
    WgArgs r{};
    r.partials = partials;
    r.B = B, r.X = X, r.Y = Y, r.Z = Z;
    r.nzc = (Z + ring::ZT - 1) / ring::ZT;
    r.zbox = Z % ring::ZT ? 64 : ring::ZT;
    CUtensorMap xm, xh, dm;
    if (!act_map(&xm, x, B, X, Y, Z, r.zbox) || !act_map(&xh, x, B, X, Y, Z, 16) || !act_map(&dm, dy, B, X, Y, Z, r.zbox))
        return cudaErrorInvalidValue;
    const int most = std::min(sms, max_ctas);
    const long long ncol = (long long)B * X * r.nzc;
    r.nseg = segments(ncol, Y, most, 1);
    if (ncol * r.nseg > (1LL << 30)) return cudaErrorInvalidValue;  // unit index would overflow int
    r.nunits = (int)(ncol * r.nseg);
    *ctas = std::min(r.nunits, most);
    cudaError_t e = cudaFuncSetAttribute(conv_wgrad_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, wg::SMEM);
    if (e != cudaSuccess) return e;
    conv_wgrad_tc_kernel<<<*ctas, wg::NTH, wg::SMEM, st>>>(xm, xh, dm, r);
    return cudaGetLastError();
}

cudaError_t tc_take_timeout(int* flag) {
    cudaError_t e = cudaMemcpyFromSymbol(flag, g_tc_timeout, sizeof(int));
    if (e != cudaSuccess || !*flag) return e;
    const int zero = 0;
    return cudaMemcpyToSymbol(g_tc_timeout, &zero, sizeof(int));
}

}  // namespace evxnn
