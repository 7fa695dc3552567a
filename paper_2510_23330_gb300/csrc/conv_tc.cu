// conv_tc.cu -- 3^3 "same" convolution of BF16 NDHWC activations on the
// 5th-generation tensor cores (tcgen05 + TMEM), used for the forward pass and
// the input gradient of the surrogate U-Net's 3^3 convolutions (Sec. 3.3 of
// Hirashima et al., SC'25).
//
// Activations are blocked by 8 channels, [batch][channel / 8][z][y][x][8], so
// 10 x voxels of one channel group are one contiguous 160-byte row.
//
// One output tile is 8 (x) x 16 (y) voxels x Zt z-planes; each z-plane is one
// M = 128 MMA row block (row r = 8 y + x).  The tile's input halo,
// (Zt + 2) x 18 x 10 voxels, is brought into shared memory once by TMA (one
// 4-D box of 18 (Zt + 2) rows of 160 bytes per channel group; out-of-range
// voxels are zero-filled by the TMA unit, which is exactly the zero padding
// of the convolution) and lands as [channel group][z][y][x][8 channels]:
// eight consecutive x voxels of one channel group form one 8 x 16-byte core
// matrix of the canonical K-major no-swizzle layout, so every one of the 27
// taps is the same descriptor with its start address shifted by the tap's
// (z, y, x) offset -- no im2col copy.
// The weights of all taps stay resident in shared memory for the whole
// persistent CTA, packed [tap][channel group][N][8].
//
// Roles (352 threads): warp 8 lane 0 issues the TMA loads, warps 9 and 10 run
// the MMA loop warp-uniformly and one elected lane of each issues tcgen05.mma
// (FP32 accumulators in TMEM; one warp when the z-taps share an MMA or the tile
// has one plane), warps 0..7 read TMEM with tcgen05.ld and apply bias, ReLU and
// the BF16 store.  Halo buffers and TMEM accumulators are double buffered where
// they fit so the loads of tile i + 1, the MMAs of tile i and the epilogue of
// tile i - 1 overlap.  Every mbarrier wait is bounded (1 s of %globaltimer); a
// wait that runs out sets the error word, all roles leave their loops, in-flight
// copies and MMAs are drained (again bounded) and TMEM is freed before the CTA
// exits.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <mutex>

#include "common.cuh"
#include "conv_tc.cuh"

typedef __nv_bfloat16 bf16;

namespace gnb {

namespace {

constexpr int EPI_WARPS = 8, TMA_WARP = 8, MMA_WARP = 9;  // then two MMA warps
constexpr int TC_THREADS = 32 * (MMA_WARP + 2);
constexpr int HX = 10, HY = 18;          // halo extent in x and y
constexpr unsigned ROW_BYTES = 16;       // one voxel of one 8-channel group
constexpr unsigned YSTRIDE = HX * ROW_BYTES;
constexpr unsigned ZSTRIDE = HY * YSTRIDE;
constexpr unsigned BIAS_AT = 256;        // after the barriers, TMEM slot and abort word
constexpr unsigned HDR = BIAS_AT + 1024; // with the bias of up to 256 output channels
constexpr int MAX_WSTAGE = 4;            // weight ring stages when the weights are streamed
constexpr unsigned ALIGN_SLACK = 1024;
constexpr unsigned long long WAIT_NS = 1000000000ull;

enum { B_W = 0, B_HF = 1, B_HE = 3, B_AF = 5, B_AE = 7, B_DR = 9, B_WF = 10, B_WE = 14, NBARS = 18 };

struct TcArgs {
    const bf16 *w;
    const float *bias;
    bf16 *out1, *out2;
    int N, K, C1, O1, relu;
    int B, D, H, W;
    int Zt, nbuf, nacc, tx, ty, tz;  // nbuf halo buffers, nacc accumulator buffers
    int wstages;  // 0: all 27 taps resident; else a ring of this many one-tap stages
    int dzn;      // 1: the three z-taps share one MMA (N = 3 N_out, sliding TMEM windows)
    unsigned acc_cols;  // TMEM columns of one accumulator buffer
    long long ntiles;
    unsigned wbytes, plane, halo, off_w, off_h, tx_bytes, tmem_cols;
    int *err;
};

__device__ __forceinline__ unsigned smem_u32(const void *p) { return (unsigned)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mb_init(unsigned bar, unsigned count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mb_expect_tx(unsigned bar, unsigned bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mb_arrive(unsigned bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(bar) : "memory");
}
__device__ __forceinline__ bool mb_try(unsigned bar, unsigned parity)
{
    unsigned ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}
__device__ __forceinline__ unsigned long long gtimer()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// Bounded wait for the phase of `parity`.  Returns false when another role
// has aborted (honour_abort) or after WAIT_NS, in which case it aborts the
// CTA and records `code` in the error word.
__device__ __noinline__ bool mb_wait(unsigned bar, unsigned parity, volatile int *abort_flag, int *err, int code,
                        bool honour_abort = true)
{
    unsigned long long t0 = 0;
    for (unsigned it = 0;; it++) {
        if (mb_try(bar, parity)) return true;
        if (honour_abort && *abort_flag) return false;
        if ((it & 31u) == 0) {
            unsigned long long t = gtimer();
            if (t0 == 0) t0 = t;
            else if (t - t0 > WAIT_NS) {
                *abort_flag = 1;
                atomicExch(err, code);
                return false;
            }
        }
    }
}

// The same with the first test inline: between the MMAs of two taps or tiles a
// call and its return cost more than the tensor core's queue covers.
__device__ __forceinline__ bool mb_wait_ready(unsigned bar, unsigned parity, volatile int *abort_flag, int *err, int code)
{
    return mb_try(bar, parity) || mb_wait(bar, parity, abort_flag, err, code);
}

__device__ __forceinline__ void tma_load_4d(unsigned dst, const CUtensorMap *m, int c0, int c1, int c2, int c3,
                                            unsigned bar)
{
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, "
        "%5}], [%6];\n" ::"r"(dst),
        "l"(reinterpret_cast<unsigned long long>(m)), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(bar)
        : "memory");
}
__device__ __forceinline__ void bulk_load(unsigned dst, const void *src, unsigned bytes, unsigned bar)
{
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n" ::"r"(dst),
                 "l"(src), "r"(bytes), "r"(bar)
                 : "memory");
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory"); }

// Shared-memory matrix descriptors, canonical K-major layout without swizzle:
// start address, leading-dimension byte offset (between core matrices along
// K), stride-dimension byte offset (between 8-row groups along M or N), and
// the descriptor version bit 46.  The low 32-bit word holds the start address
// in 16-byte units (bits 0-13) and the leading offset (bits 16-29), so moving
// the start by a multiple of 16 bytes is one add on the low word; the high
// word holds the stride offset and the version bit.
__device__ __forceinline__ unsigned sdesc_lo(unsigned addr, unsigned lbo)
{
    return ((addr & 0x3FFFFu) >> 4) | ((lbo >> 4) << 16);
}
__device__ __forceinline__ unsigned sdesc_hi(unsigned sbo) { return (sbo >> 4) | (1u << 14); }
__device__ __forceinline__ unsigned long long dpair(unsigned lo, unsigned hi)
{
    return ((unsigned long long)hi << 32) | lo;
}

// MMA and commit are executed by the whole warp in uniform control flow (so
// the operands stay warp-uniform); elect.sync picks the one lane that issues.
__device__ __forceinline__ void tc_mma_elect(unsigned d, unsigned long long a, unsigned long long b, unsigned idesc,
                                             unsigned acc)
{
    asm volatile(
        "{\n .reg .pred e, p;\n elect.sync _|e, 0xffffffff;\n setp.ne.b32 p, %4, 0;\n"
        " @e tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d),
        "l"(a), "l"(b), "r"(idesc), "r"(acc)
        : "memory");
}
__device__ __forceinline__ void tc_commit_elect(unsigned bar)
{
    asm volatile(
        "{\n .reg .pred e;\n elect.sync _|e, 0xffffffff;\n"
        " @e tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n}\n" ::"r"(bar)
        : "memory");
}

// NC consecutive FP32 columns of this thread's TMEM lane; the wait is in the
// same statement so no use of the registers can be scheduled before it.
template <int NC>
__device__ void tc_ld(unsigned taddr, unsigned *r);
template <>
__device__ __forceinline__ void tc_ld<16>(unsigned taddr, unsigned *r)
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, "
                 "%13, %14, %15}, [%16];\n"
                 "tcgen05.wait::ld.sync.aligned;\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]),
                   "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]),
                   "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
                 : "r"(taddr)
                 : "memory");
}
template <>
__device__ __forceinline__ void tc_ld<32>(unsigned taddr, unsigned *r)
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, "
                 "%13, %14, %15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31},"
                 " [%32];\n"
                 "tcgen05.wait::ld.sync.aligned;\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]),
                   "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]),
                   "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]),
                   "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
                   "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]),
                   "=r"(r[30]), "=r"(r[31])
                 : "r"(taddr)
                 : "memory");
}
__device__ __forceinline__ void tc_ld16(unsigned taddr, float *v)
{
    unsigned r[16];
    tc_ld<16>(taddr, r);
#pragma unroll
    for (int i = 0; i < 16; i++) v[i] = __uint_as_float(r[i]);
}

// 8 consecutive FP32 columns of this thread's TMEM lane.
__device__ __forceinline__ void tc_ld8(unsigned taddr, float *v)
{
    unsigned r[8];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];\n"
        "tcgen05.wait::ld.sync.aligned;\n"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
        : "r"(taddr)
        : "memory");
#pragma unroll
    for (int i = 0; i < 8; i++) v[i] = __uint_as_float(r[i]);
}

__device__ __forceinline__ void decode_tile(const TcArgs &p, int Zt, long long t, int &bb, int &z0, int &y0, int &x0)
{
    int xt = (int)(t % p.tx);
    t /= p.tx;
    int yt = (int)(t % p.ty);
    t /= p.ty;
    int zt = (int)(t % p.tz);
    bb = (int)(t / p.tz);
    x0 = 8 * xt;
    y0 = 16 * yt;
    z0 = Zt * zt;
}

// kind::f16 instruction descriptor without N: FP32 accumulator (bit 4), BF16 A
// (bits 7-9 = 1) and B (bits 10-12 = 1), both K-major, M >> 4 at bit 24
// (M = 128); N >> 3 goes to bit 17.
constexpr unsigned IDESC0 = (1u << 4) | (1u << 7) | (1u << 10) | ((128u >> 4) << 24);

// Bytes of one channel group of a tile's halo.
__host__ __device__ constexpr unsigned plane_bytes(int zt) { return ((unsigned)(zt + 2) * ZSTRIDE + 127u) & ~127u; }

// The tensor core needs max(N / 2, 32 + N / 4) cycles for one 128 x N x 16 MMA
// (measured; the 4 KB of A and the 32 N bytes of B come from shared memory at
// 128 bytes a cycle), whatever the accumulator, the start address or the
// stride: 44 at N = 48, 48 at N = 64, 56 at N = 96.  One warp issues that fast
// only when every operand is a loop-carried base plus a compile-time constant;
// with N, the plane size or K read from the arguments, and 64-bit divisions by
// the ring size between the taps, an MMA took 71 (resident weights) to 98
// (streamed) cycles at N = 64.  So the tile depth, N and the K steps of a block are
// template parameters; 0 stands for a run-time value.

// The MMAs of one dz-in-N tile.  Input plane j, in-plane tap (ty, tx): one
// MMA whose columns are output planes j - 2, j - 1, j (z-taps 2, 1, 0), less
// those outside the tile.  Windows of planes j = r, r + 3, ... are disjoint, so
// every output sums its z-taps in the order of r and, within one, (ty, tx) and
// the channels in order; those of r = 0 cover every output plane, so its first
// MMAs start the sums.
template <int ZT, int NKS, int NN>
__device__ __forceinline__ void issue_dzn(const TcArgs &p, unsigned alo0, unsigned sW, unsigned d0)
{
    const int Zt = ZT ? ZT : p.Zt, nks = NKS ? NKS : (p.K >> 4), N = NN ? NN : p.N;
    const unsigned ahi = sdesc_hi(YSTRIDE), bhi = sdesc_hi(128u);
    const unsigned zs4 = ZSTRIDE >> 4, pl4 = (2u * plane_bytes(Zt)) >> 4;
    const unsigned n3 = 3u * (unsigned)N;
    const unsigned wyx4 = ((unsigned)nks * 2u * n3 * 16u) >> 4;  // one (ty, tx) slice of weights
    const unsigned bk4 = (2u * n3 * 16u) >> 4;
    const unsigned blo0 = sdesc_lo(sW, n3 * 16u);
#pragma unroll
    for (int r = 0; r < 3; r++)
#pragma unroll
        for (int yx = 0; yx < 9; yx++) {
            const unsigned aoff = ((unsigned)(yx / 3) * YSTRIDE + (unsigned)(yx % 3) * ROW_BYTES) >> 4;
#pragma unroll
            for (int ks = 0; ks < nks; ks++)
#pragma unroll
                for (int j = r; j < Zt + 2; j += 3) {
                    const int q0 = j < 2 ? 2 - j : 0, q1 = j < Zt ? 3 : Zt + 2 - j;  // z-tap blocks inside the tile
                    tc_mma_elect(d0 + (unsigned)((j - 2 + q0) * N),
                                 dpair(alo0 + aoff + (unsigned)ks * pl4 + (unsigned)j * zs4, ahi),
                                 dpair(blo0 + (unsigned)yx * wyx4 + (unsigned)ks * bk4 + (unsigned)(q0 * N), bhi),
                                 IDESC0 | ((unsigned)((q1 - q0) * N >> 3) << 17), (unsigned)(r + yx + ks != 0));
                }
        }
}

// The MMAs of TAPS consecutive x-taps of one plain tile: per K step (innermost,
// so every accumulator sums its taps and channels in one fixed order) one MMA
// for each of this warp's z-planes, in blocks of NKS K steps.  FIRST: the first MMA
// of each plane starts its sum.
template <int ZT, int NKS, int NN, int TAPS, bool FIRST>
__device__ __forceinline__ void issue_taps(const TcArgs &p, unsigned alo, unsigned blo, unsigned d0, int mw)
{
    constexpr int U = NKS ? NKS : 1;
    const int Zt = ZT ? ZT : p.Zt, blocks = (p.K >> 4) / U, N = NN ? NN : p.N, nmma = Zt > 1 ? 2 : 1;
    alo += (unsigned)mw * (ZSTRIDE >> 4);  // planes mw, mw + 2, ...
    d0 += (unsigned)(mw * N);
    const unsigned ahi = sdesc_hi(YSTRIDE), bhi = sdesc_hi(128u);
    const unsigned zs4 = ZSTRIDE >> 4, pl4 = (2u * plane_bytes(Zt)) >> 4, nb4 = (2u * (unsigned)N * 16u) >> 4;
    const unsigned idesc = IDESC0 | ((unsigned)(N >> 3) << 17);
#pragma unroll
    for (int t = 0; t < TAPS; t++) {
        unsigned at = alo + (unsigned)t * (ROW_BYTES >> 4);
#pragma unroll 1
        for (int kb = 0; kb < blocks; kb++, at += U * pl4, blo += U * nb4) {
#pragma unroll
            for (int u = 0; u < U; u++)
#pragma unroll
                for (int zz = 0; zz < Zt - (ZT ? 0 : mw); zz += nmma)
                    tc_mma_elect(d0 + (unsigned)(zz * N), dpair(at + (unsigned)u * pl4 + (unsigned)zz * zs4, ahi),
                                 dpair(blo + (unsigned)u * nb4, bhi), idesc,
                                 FIRST && t == 0 && u == 0 ? (unsigned)(kb != 0) : 1u);
        }
    }
}

// DZ: 1 dz-in-N, 0 plain, -1 read from p; ZT: tile depth (0: read from p);
// NKS: K / 16 (plain tiles: the K steps of one straight-line block; 0: read from p);
// NN: the output channels (0: read from p).
// CTAs that can share an SM: the registers are limited for two where the shared
// memory of a dz-in-N tile admits two (32 -> 16 channels, one CTA: 285 us
// without the limit on 32 x 64^3 voxels, 355 with it; 16 -> 32 channels on
// 32 x 32^3, two CTAs: 38 us with one, 29 with two).
__host__ __device__ constexpr int tc_min_ctas(int dz, int zt, int nks, int nn)
{
    return dz == 1 && zt && 27u * (unsigned)(nn * nks) * 32u + 4u * (unsigned)nks * plane_bytes(zt) > TC_SMEM_SM / 2u ? 1 : 2;
}

template <int DZ, int ZT, int NKS, int NN>
__global__ void __launch_bounds__(TC_THREADS, tc_min_ctas(DZ, ZT, NKS, NN))
    k_conv3_tc(const __grid_constant__ CUtensorMap m1, const __grid_constant__ CUtensorMap m2, const TcArgs p)
{
    const int Zt = ZT ? ZT : p.Zt;
    const bool dzn = DZ >= 0 ? DZ != 0 : p.dzn != 0;
    extern __shared__ unsigned char dsm[];
    const unsigned raw = smem_u32(dsm);
    const unsigned sb = (raw + (ALIGN_SLACK - 1)) & ~(ALIGN_SLACK - 1);
    unsigned char *gb = dsm + (sb - raw);
    unsigned *slot = reinterpret_cast<unsigned *>(gb + 8 * NBARS);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(gb + 8 * NBARS + 4);
    const unsigned sW = sb + p.off_w, sH = sb + p.off_h;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    auto bar = [&](int i) { return sb + 8u * (unsigned)i; };

    // plain tiles of two and more planes are issued by two warps, each with its
    // share of the planes (the accumulators are independent): one warp spent
    // 60 to 90 cycles per 48-cycle MMA (N = 64) on the waits and commits of a tap
    const int nmma = !dzn && Zt > 1 ? 2 : 1;
    if (threadIdx.x == 0) {
        mb_init(bar(B_W), 1);
        for (int b = 0; b < 2; b++) {
            mb_init(bar(B_HF + b), 1);
            mb_init(bar(B_HE + b), (unsigned)nmma);
            mb_init(bar(B_AF + b), (unsigned)nmma);
            mb_init(bar(B_AE + b), 32 * EPI_WARPS);
        }
        mb_init(bar(B_DR), (unsigned)nmma);
        for (int q = 0; q < MAX_WSTAGE; q++) {
            mb_init(bar(B_WF + q), 1);
            mb_init(bar(B_WE + q), (unsigned)nmma);
        }
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    float *sbias = reinterpret_cast<float *>(gb + BIAS_AT);
    if (p.bias)
        for (int n = threadIdx.x; n < p.N; n += TC_THREADS) sbias[n] = p.bias[n];
    if (warp == TMA_WARP) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_u32(slot)),
                     "r"(p.tmem_cols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const unsigned tmem = *slot;
    const int kc8 = p.K >> 3;
    if (warp == TMA_WARP) {
        if (lane == 0) {
            // ---------------------------------------------------------- producer
            const unsigned wtap = (unsigned)kc8 * (unsigned)p.N * 16u;  // bytes of one tap's weights
            if (!p.wstages) {
                mb_expect_tx(bar(B_W), p.wbytes);
                for (unsigned o = 0; o < p.wbytes; o += 32768u) {
                    unsigned n = p.wbytes - o < 32768u ? p.wbytes - o : 32768u;
                    bulk_load(sW + o, reinterpret_cast<const unsigned char *>(p.w) + o, n, bar(B_W));
                }
            }
            int uses[2] = {0, 0};
            // the weight ring: the next stage and how often it was filled (counted,
            // as 64-bit divisions by the ring size took as long as a tap's MMAs)
            int st = 0;
            unsigned round = 0;
            bool stop = false;
            int i = 0;
            for (long long t = blockIdx.x; t < p.ntiles; t += gridDim.x, i++) {
                const int b = i % p.nbuf;
                const unsigned k = (unsigned)(i / p.nbuf);
                if (k > 0 && !mb_wait(bar(B_HE + b), (k - 1) & 1u, abort_flag, p.err, 1)) break;
                int bb, z0, y0, x0;
                decode_tile(p, Zt, t, bb, z0, y0, x0);
                mb_expect_tx(bar(B_HF + b), p.tx_bytes);
                const unsigned dst = sH + (unsigned)b * p.halo;
                // x and the 8 channels of a group form the innermost TMA
                // dimension: start 8 (x0 - 1) elements = 16 (x0 - 1) bytes
                const int g1 = p.C1 >> 3, g2 = (p.K - p.C1) >> 3;
                for (int kc = 0; kc < kc8; kc++) {
                    if (kc < g1)
                        tma_load_4d(dst + kc * p.plane, &m1, 8 * (x0 - 1), y0 - 1, z0 - 1, bb * g1 + kc, bar(B_HF + b));
                    else
                        tma_load_4d(dst + kc * p.plane, &m2, 8 * (x0 - 1), y0 - 1, z0 - 1, bb * g2 + (kc - g1),
                                    bar(B_HF + b));
                }
                uses[b]++;
                // streamed weights: the 27 taps of this tile through the ring
                for (int tap = 0; p.wstages && tap < 27; tap++) {
                    if (round > 0 && !mb_wait(bar(B_WE + st), (round - 1) & 1u, abort_flag, p.err, 8)) {
                        stop = true;
                        break;
                    }
                    mb_expect_tx(bar(B_WF + st), wtap);
                    bulk_load(sW + (unsigned)st * wtap, reinterpret_cast<const unsigned char *>(p.w) + (size_t)tap * wtap,
                              wtap, bar(B_WF + st));
                    if (++st == p.wstages) { st = 0; round++; }
                }
                if (stop) break;
            }
            // drain: every copy this CTA issued has landed before it exits
            if (!p.wstages) mb_wait(bar(B_W), 0, abort_flag, p.err, 2, false);
            for (int b = 0; b < 2; b++)
                if (uses[b] > 0) mb_wait(bar(B_HF + b), (unsigned)(uses[b] - 1) & 1u, abort_flag, p.err, 2, false);
            for (int q = 0; q < p.wstages; q++) {
                const unsigned fills = round + (q < st ? 1u : 0u);
                if (fills > 0) mb_wait(bar(B_WF + q), (fills - 1) & 1u, abort_flag, p.err, 2, false);
            }
        }
    } else if (warp >= MMA_WARP) {
        const int mw = warp - MMA_WARP;
        // ------------------------------------------------------------------ MMA
        // The Zt z-planes of a tile accumulate into Zt independent TMEM
        // blocks; their MMAs are interleaved so consecutive MMAs never feed
        // the same accumulator.
        int ok = mw >= nmma ? 0 : (p.wstages ? 1 : mb_wait(bar(B_W), 0, abort_flag, p.err, 3));
        if (__all_sync(0xffffffffu, ok)) {
            const long long first_reuse = blockIdx.x + (long long)p.nacc * gridDim.x;
            int st = 0;  // the weight ring's next stage and the parity of its fill
            unsigned wpar = 0;
            const unsigned wtap = (unsigned)kc8 * (unsigned)p.N * 16u;  // bytes of one tap's weights
            const unsigned nbytes16 = (unsigned)p.N * 16u;              // one channel group of weights
            int b = 0, ab = 0;  // halo and accumulator buffer, and the parities of their barriers' phases
            unsigned hpar = 0, apar = 1;
            for (long long t = blockIdx.x; t < p.ntiles; t += gridDim.x) {
                ok = mb_wait_ready(bar(B_HF + b), hpar, abort_flag, p.err, 4);
                if (t >= first_reuse) ok = ok && mb_wait_ready(bar(B_AE + ab), apar, abort_flag, p.err, 5);
                if (!__all_sync(0xffffffffu, ok)) break;
                tc_fence_after();
                const unsigned hb = sH + (unsigned)b * p.halo;
                const unsigned d0 = tmem + (unsigned)ab * p.acc_cols;
                bool stop = false;
                // descriptors are stepped as 32-bit low words (start address in
                // 16-byte units): a few adds per MMA
                const unsigned alo0 = sdesc_lo(hb, p.plane);
                if (dzn) issue_dzn<ZT, NKS, NN>(p, alo0, sW, d0);
                for (int row = 0; !dzn && row < 9; row++) {  // (tz, ty); the three tx inside
                    const unsigned alo = alo0 + (((unsigned)(row / 3) * ZSTRIDE + (unsigned)(row % 3) * YSTRIDE) >> 4);
                    if (!p.wstages) {
                        const unsigned blo = sdesc_lo(sW + 3u * (unsigned)row * wtap, nbytes16);
                        if (row) issue_taps<ZT, NKS, NN, 3, false>(p, alo, blo, d0, mw);
                        else issue_taps<ZT, NKS, NN, 3, true>(p, alo, blo, d0, mw);
                        continue;
                    }
                    for (int tx = 0; tx < 3; tx++) {
                        ok = mb_wait_ready(bar(B_WF + st), wpar, abort_flag, p.err, 9);
                        if (!__all_sync(0xffffffffu, ok)) { stop = true; break; }
                        tc_fence_after();
                        const unsigned at = alo + (unsigned)tx * (ROW_BYTES >> 4);
                        const unsigned blo = sdesc_lo(sW + (unsigned)st * wtap, nbytes16);
                        if (row + tx) issue_taps<ZT, NKS, NN, 1, false>(p, at, blo, d0, mw);
                        else issue_taps<ZT, NKS, NN, 1, true>(p, at, blo, d0, mw);
                        tc_commit_elect(bar(B_WE + st));  // the stage is free once these MMAs complete
                        if (++st == p.wstages) { st = 0; wpar ^= 1u; }
                    }
                    if (stop) break;
                }
                if (stop) break;
                tc_commit_elect(bar(B_HE + b));
                tc_commit_elect(bar(B_AF + ab));
                if (++b == p.nbuf) { b = 0; hpar ^= 1u; }
                if (++ab == p.nacc) { ab = 0; apar ^= 1u; }
            }
        }
        // drain: all MMAs issued by the MMA warps' elected lanes are complete
        if (mw < nmma) {
            tc_commit_elect(bar(B_DR));
            mb_wait(bar(B_DR), 0, abort_flag, p.err, 6, false);
        }
        __syncwarp();
    } else {
        // ------------------------------------------------------------ epilogue
        // The accumulators' columns are plane-major; each of the two warps of a
        // lane quarter reads every other CH of them.  Bias, ReLU, conversion
        // and stores are one warp's serial instructions: with one warp per
        // quarter the 16-channel layers waited for them (4500 of a tile's 5500
        // cycles).  A buffer is handed back before its last columns are stored.
        constexpr int COLS = ZT * NN, CH = COLS >= 64 ? 32 : 16;
        static_assert(COLS % CH == 0, "columns are read in whole chunks");
        const int N = NN ? NN : p.N;
        const int r = 32 * (warp & 3) + lane;  // TMEM lane = row of the M = 128 block
        const unsigned lane_addr = (unsigned)(32 * (warp & 3)) << 16;
        const long long Vs = (long long)p.D * p.H * p.W;
        const int HW = p.H * p.W;
        int i = 0;
        for (long long t = blockIdx.x; t < p.ntiles; t += gridDim.x, i++) {
            const int b = i % p.nacc;
            const unsigned k = (unsigned)(i / p.nacc);
            int ok = mb_wait(bar(B_AF + b), k & 1u, abort_flag, p.err, 7);
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) break;
            tc_fence_after();
            int bb, z0, y0, x0;
            decode_tile(p, Zt, t, bb, z0, y0, x0);
            const int x = x0 + (r & 7), y = y0 + (r >> 3);
            const bool inxy = x < p.W && y < p.H;
            const long long sv0 = ((long long)z0 * p.H + y) * p.W + x;
            const int cols = Zt * N;
            if ((warp >> 2) * CH >= cols) {
                tc_fence_before();
                mb_arrive(bar(B_AE + b));
            }
#pragma unroll 1
            for (int c = (warp >> 2) * CH; c < cols; c += 2 * CH) {
                unsigned u[CH];
                __syncwarp();
                tc_ld<CH>(tmem + lane_addr + (unsigned)b * p.acc_cols + (unsigned)c, u);
                if (c + 2 * CH >= cols) {
                    tc_fence_before();
                    mb_arrive(bar(B_AE + b));
                }
#pragma unroll
                for (int g = 0; g < CH; g += 16) {
                    const int zz = (c + g) / N, c0 = (c + g) % N;
                    if (!inxy || z0 + zz >= p.D) continue;
                    float f[16];
#pragma unroll
                    for (int q = 0; q < 16; q++) f[q] = __uint_as_float(u[g + q]);
                    if (p.bias) {
#pragma unroll
                        for (int q = 0; q < 16; q += 4) {
                            const float4 bq = *reinterpret_cast<const float4 *>(sbias + c0 + q);
                            f[q] += bq.x; f[q + 1] += bq.y; f[q + 2] += bq.z; f[q + 3] += bq.w;
                        }
                    }
                    if (p.relu) {
#pragma unroll
                        for (int q = 0; q < 16; q++) f[q] = fmaxf(f[q], 0.f);
                    }
                    uint4 o[2];
                    unsigned *ou = reinterpret_cast<unsigned *>(o);
#pragma unroll
                    for (int q = 0; q < 8; q++) {
                        __nv_bfloat162 h2 = __floats2bfloat162_rn(f[2 * q], f[2 * q + 1]);
                        ou[q] = *reinterpret_cast<unsigned *>(&h2);
                    }
                    // two channel groups: two 16-byte pieces, Vs * 8 elements apart
                    const bool lo = c0 < p.O1;
                    const int Cx = lo ? p.O1 : N - p.O1, cc = lo ? c0 : c0 - p.O1;
                    bf16 *dst = (lo ? p.out1 : p.out2) +
                                (((long long)bb * (Cx >> 3) + (cc >> 3)) * Vs + sv0 + (long long)zz * HW) * 8;
                    *reinterpret_cast<uint4 *>(dst) = o[0];
                    *reinterpret_cast<uint4 *>(dst + Vs * 8) = o[1];
                }
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == TMA_WARP) {
        __syncwarp();
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(p.tmem_cols)
                     : "memory");
    }
}

typedef CUresult (*encode_fn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                              const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                              CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

encode_fn get_encode()
{
    static encode_fn fn = []() -> encode_fn {
        void *f = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000, cudaEnableDefault, &q) !=
                cudaSuccess ||
            q != cudaDriverEntryPointSuccess) {
            cudaGetLastError();
            return nullptr;
        }
        return reinterpret_cast<encode_fn>(f);
    }();
    return fn;
}

// Tensor map of a blocked BF16 tensor [B][C / 8][D][H][W][8] viewed as 4-D
// (8 W, H, D, B C / 8) and read in halo boxes of 8 x 10 elements (10 voxels
// of one channel group) x 18 x zh.
bool make_map(CUtensorMap *m, const bf16 *ptr, int C, int B, int D, int H, int W, int zh)
{
    encode_fn enc = get_encode();
    if (!enc) return false;
    cuuint64_t dims[4] = {(cuuint64_t)W * 8, (cuuint64_t)H, (cuuint64_t)D, (cuuint64_t)B * (C / 8)};
    cuuint64_t strides[3] = {(cuuint64_t)W * 16, (cuuint64_t)H * W * 16, (cuuint64_t)D * H * W * 16};
    cuuint32_t box[4] = {8 * HX, (cuuint32_t)HY, (cuuint32_t)zh, 1};
    cuuint32_t es[4] = {1, 1, 1, 1};
    return enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<bf16 *>(ptr), dims, strides, box, es,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

int device_sms()
{
    static int n = []() {
        int d = 0, v = 0;
        cudaGetDevice(&d);
        cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, d);
        return v > 0 ? v : 1;
    }();
    return n;
}

unsigned pow2_at_least(unsigned v)
{
    unsigned c = 32;
    while (c < v) c <<= 1;
    return c;
}


// ------------------------------------------------------------------ UP2
// 2x2x2 transposed convolution with stride 2 on the tensor cores: one tile is
// 128 consecutive coarse voxels of one batch entry (M = 128) and all eight
// taps' output channels form N = 8 N_out, so a tile is K / 16 MMAs (split in
// two when 8 N_out > 256).  In the blocked layout the 128 voxels of one
// channel group are 2 KB of contiguous memory, i.e. exactly a column of
// K-major core matrices; the tile and the weights arrive by bulk copies.
struct Up2Args {
    const bf16 *in;      // coarse [B][K / 8][Vc][8]
    const bf16 *w;       // [K / 8][8 N][8], row t N + n = tap t, output channel n
    const float *bias;   // [N] or null
    bf16 *out;           // fine [B][N / 8][8 Vc][8]
    int K, N, Dc;        // input channels, output channels, coarse grid edge
    long long Vc, ntiles;
    unsigned abytes, wbytes, tmem_cols, idesc, nsplit, ncols_split;
    int *err;
};
constexpr unsigned UP_HDR = 256;

__global__ void __launch_bounds__(128) k_up2_tc(const Up2Args p)
{
    extern __shared__ unsigned char dsm[];
    const unsigned raw = smem_u32(dsm);
    const unsigned sb = (raw + (ALIGN_SLACK - 1)) & ~(ALIGN_SLACK - 1);
    unsigned char *gb = dsm + (sb - raw);
    unsigned *slot = reinterpret_cast<unsigned *>(gb + 16);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(gb + 20);
    const unsigned bar_ld = sb, bar_mma = sb + 8;
    const unsigned sA = sb + UP_HDR, sB = sA + p.abytes;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const long long r0 = (long long)blockIdx.x * 128;
    const long long bb = r0 / p.Vc, v0 = r0 - bb * p.Vc;
    const int kc8 = p.K >> 3;
    if (threadIdx.x == 0) {
        mb_init(bar_ld, 1);
        mb_init(bar_mma, 1);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_u32(slot)),
                     "r"(p.tmem_cols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const unsigned tmem = *slot;
    if (threadIdx.x == 0) {
        mb_expect_tx(bar_ld, p.abytes + p.wbytes);
        for (int kc = 0; kc < kc8; kc++)
            bulk_load(sA + (unsigned)kc * 2048u, p.in + ((bb * kc8 + kc) * p.Vc + v0) * 8, 2048u, bar_ld);
        for (unsigned o = 0; o < p.wbytes; o += 32768u) {
            unsigned n = p.wbytes - o < 32768u ? p.wbytes - o : 32768u;
            bulk_load(sB + o, reinterpret_cast<const unsigned char *>(p.w) + o, n, bar_ld);
        }
    }
    bool ok = true;
    if (warp == 1) {
        ok = __all_sync(0xffffffffu, mb_wait(bar_ld, 0, abort_flag, p.err, 11));
        if (ok) {
            tc_fence_after();
            const unsigned ahi = sdesc_hi(128u), bhi = sdesc_hi(128u);
            const unsigned nrow16 = (unsigned)(8 * p.N) * 16u;  // one channel group of all weight rows
            for (int ks = 0; ks < (p.K >> 4); ks++)
                for (unsigned h = 0; h < p.nsplit; h++)
                    tc_mma_elect(tmem + h * p.ncols_split,
                                 dpair(sdesc_lo(sA + (unsigned)ks * 4096u, 2048u), ahi),
                                 dpair(sdesc_lo(sB + (unsigned)ks * 2u * nrow16 + h * p.ncols_split * 16u, nrow16), bhi),
                                 p.idesc, ks != 0);
            tc_commit_elect(bar_mma);
        }
    }
    // every thread: the accumulators are ready (or the CTA gave up)
    ok = mb_wait(bar_mma, 0, abort_flag, p.err, 12);
    ok = __all_sync(0xffffffffu, ok);
    if (ok) {
        tc_fence_after();
        const int r = 32 * warp + lane;
        const unsigned lane_addr = (unsigned)(32 * warp) << 16;
        const long long v = v0 + r;
        const int D = p.Dc, x = (int)(v % D), y = (int)((v / D) % D), z = (int)(v / ((long long)D * D));
        const long long Vf = 8 * p.Vc;
        const int F = 2 * D;
        // taps in pairs (dx = 0, 1): the two fine voxels are adjacent in x,
        // so each channel group is one 32-byte store
        for (int tp = 0; tp < 4; tp++) {
            const int dz = tp >> 1, dy = tp & 1;
            const long long fv = ((long long)(2 * z + dz) * F + (2 * y + dy)) * F + 2 * x;
            for (int g = 0; g < (p.N >> 3); g++) {
                float f0[16], f1[16];
                // columns of tap (dz, dy, 0) and (dz, dy, 1): t N + 8 g + j
                const unsigned c0 = (unsigned)((2 * tp) * p.N + 8 * g), c1 = c0 + (unsigned)p.N;
                __syncwarp();
                tc_ld8(tmem + lane_addr + c0, f0);
                tc_ld8(tmem + lane_addr + c1, f1);
                uint4 o[2];
                unsigned *ou = reinterpret_cast<unsigned *>(o);
#pragma unroll
                for (int q = 0; q < 4; q++) {
                    const float b0 = p.bias ? __ldg(p.bias + 8 * g + 2 * q) : 0.f;
                    const float b1 = p.bias ? __ldg(p.bias + 8 * g + 2 * q + 1) : 0.f;
                    __nv_bfloat162 h0 = __floats2bfloat162_rn(f0[2 * q] + b0, f0[2 * q + 1] + b1);
                    __nv_bfloat162 h1 = __floats2bfloat162_rn(f1[2 * q] + b0, f1[2 * q + 1] + b1);
                    ou[q] = *reinterpret_cast<unsigned *>(&h0);
                    ou[4 + q] = *reinterpret_cast<unsigned *>(&h1);
                }
                bf16 *dst = p.out + ((bb * (p.N >> 3) + g) * Vf + fv) * 8;
                reinterpret_cast<uint4 *>(dst)[0] = o[0];
                reinterpret_cast<uint4 *>(dst)[1] = o[1];
            }
        }
    }
    if (threadIdx.x == 0) mb_wait(bar_ld, 0, abort_flag, p.err, 13, false);  // no copy outlives the CTA
    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(p.tmem_cols)
                     : "memory");
    }
}


// ------------------------------------------------------------------ WGRAD
// Weight gradient of a 3^3 "same" convolution on the tensor cores:
//   dW[t][c][n] = sum_v x(v + tap t)[c] * g(v)[n]
// as a GEMM whose M = 128 rows are (tap slot s, input channel c) pairs --
// 128 / C taps of one tap group side by side, so every row is a real weight
// even for C = 16 -- whose N columns are the output channels and whose K is
// the voxels.  A CTA takes one tap group and one chunk of voxels.  Both
// operands are MN-major: a voxel's 8 channels are one 16-byte row of a core
// matrix (8 voxels x 8 channels, 128 bytes), which is how the blocked tensors
// hold them, so a stage of 64 voxels is filled by 16-byte asynchronous copies
// (zero-filled outside the grid) with no transposition through registers;
// each thread owns one voxel of the stage and steps its coordinates once.
// One elected lane issues four K = 16 MMAs per stage into a TMEM accumulator;
// three stage buffers, two stages of copies in flight.  At the end each warp
// reads its 32 TMEM lanes (rows) and adds them to dW with FP32 vector
// reductions (the voxel chunks are split-K).  It is bound by the instructions
// that address the copies (27 shifted 16-byte pieces per voxel and channel
// group, each with its bounds test: 56 % issue-active on a 16-channel 64^3
// layer, where L1 is at 15 %, L2 at 22 and the tensor pipe at 2.5).  All 14
// layers of a 64^3 training step (cold cache): 1,824 us with 2-byte transposing
// stores and 64-bit divisions per piece, 505 us so.
struct WgTcArgs {
    const bf16 *x1, *x2;   // input channels [0, C1) from x1, [C1, C) from x2; blocked [B][C/8][V][8]
    int C1, C;
    const bf16 *g;         // output gradient, blocked with Cg channels
    int Cg, N, Cw;         // channels of g, output channels of dW, input channels of dW (<= C)
    float *dw;             // [27][Cw][N]
    int B, D;              // grid (cube of edge D) and batch
    int ntap;              // taps per group: 128 / C
    long long V, chunk;    // voxels in all, voxels per CTA (multiple of 64)
    int nchunk;
    unsigned tmem_cols, idesc, abytes, bbytes;
    int *err;
};
constexpr unsigned WG_HDR = 256;
constexpr int WG_VS = 64;  // voxels per stage

__device__ __forceinline__ void fence_proxy_async_smem()
{
    asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
}

constexpr int WG_ST = 3;   // stage buffers

// 16-byte copy to shared memory, or zeros
__device__ __forceinline__ void cp16z(unsigned dst, const void *src, bool have)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(dst), "l"(src), "r"(have ? 16 : 0) : "memory");
}
__device__ __forceinline__ void red_v4_f32(float *a, float x, float y, float z, float w)
{
    asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};\n" ::"l"(a), "f"(x), "f"(y), "f"(z), "f"(w) : "memory");
}

__global__ void __launch_bounds__(128) k_wgrad_tc(const WgTcArgs p)
{
    extern __shared__ unsigned char dsm[];
    const unsigned raw = smem_u32(dsm);
    const unsigned sb = (raw + (ALIGN_SLACK - 1)) & ~(ALIGN_SLACK - 1);
    unsigned char *gb = dsm + (sb - raw);
    unsigned *slot = reinterpret_cast<unsigned *>(gb + 32);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(gb + 36);
    const unsigned stage_bytes = p.abytes + p.bbytes;
    unsigned char *stg = gb + WG_HDR;
    const unsigned sStg = sb + WG_HDR;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int tg = blockIdx.y;                // tap group
    const int t0 = tg * p.ntap;
    const int ntap = min(p.ntap, 27 - t0);
    const long long r0 = (long long)blockIdx.x * p.chunk, r1 = min(p.V, r0 + p.chunk);
    const int nstage = (int)((r1 - r0 + WG_VS - 1) / WG_VS);
    const int D = p.D, Vs = D * D * D;
    if (tid == 0) {
        for (int k = 0; k < WG_ST; k++) mb_init(sb + 8u * k, 1);  // commit barriers of the stage buffers
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_u32(slot)),
                     "r"(p.tmem_cols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const unsigned tmem = *slot;
    // rows of tap slots beyond ntap (a short last group) stay zero: cleared once
    for (unsigned o = (unsigned)tid * 16u; o < (unsigned)WG_ST * stage_bytes; o += 128u * 16u)
        *reinterpret_cast<uint4 *>(stg + o) = make_uint4(0u, 0u, 0u, 0u);
    __syncthreads();
    const int cg8 = p.C >> 3, ng8 = p.N >> 3, c18 = p.C1 >> 3;
    // this thread's voxel of a stage (k) and its share of the pieces (half)
    const int k = tid & (WG_VS - 1), half = tid >> 6;
    long long v = r0 + k;
    long long bb = v / Vs;
    int rem = (int)(v - bb * Vs);
    const unsigned koff = (unsigned)(k & 7) * 16u;
    const unsigned ka = (unsigned)(k >> 3) * 2048u + koff, kb = (unsigned)(k >> 3) * (unsigned)p.N * 16u + koff;
    auto load = [&](int st) {  // copies of stage st (called for st = 0, 1, 2, ... in order)
        const unsigned sA = sStg + (unsigned)(st % WG_ST) * stage_bytes, sB = sA + p.abytes;
        const bool in = v < r1;
        const int z = rem / (D * D), yx = rem - z * D * D, y = yx / D, x = yx - y * D;
        const bf16 *x1 = p.x1 + ((size_t)bb * c18 * Vs + rem) * 8;
        const bf16 *x2 = p.x2 + ((size_t)bb * (cg8 - c18) * Vs + rem) * 8;
        for (int s = 0; s < ntap; s++) {
            const int t = t0 + s, dz = t / 9 - 1, dy = (t / 3) % 3 - 1, dx = t % 3 - 1;
            const bool have = in && (unsigned)(z + dz) < (unsigned)D && (unsigned)(y + dy) < (unsigned)D &&
                              (unsigned)(x + dx) < (unsigned)D;
            const int off = have ? ((dz * D + dy) * D + dx) * 8 : 0;
            for (int cg = half; cg < cg8; cg += 2) {
                const bf16 *src = cg < c18 ? x1 + (size_t)cg * Vs * 8 : x2 + (size_t)(cg - c18) * Vs * 8;
                cp16z(sA + ka + (unsigned)(s * cg8 + cg) * 128u, have ? src + off : p.x1, have);
            }
        }
        const bf16 *g = p.g + ((size_t)bb * (p.Cg >> 3) * Vs + rem) * 8;
        for (int ng = half; ng < ng8; ng += 2) cp16z(sB + kb + (unsigned)ng * 128u, in ? g + (size_t)ng * Vs * 8 : p.g, in);
        asm volatile("cp.async.commit_group;\n" ::: "memory");
        v += WG_VS;
        rem += WG_VS;
        while (rem >= Vs) {
            rem -= Vs;
            bb++;
        }
    };
    load(0);
    if (nstage > 1) load(1);
    else asm volatile("cp.async.commit_group;\n" ::: "memory");
    bool ok = true;
    int issued = -1;  // the last stage whose MMAs were issued
    for (int st = 0; st < nstage; st++) {
        asm volatile("cp.async.wait_group 1;\n" ::: "memory");  // stage st has landed
        fence_proxy_async_smem();  // ... and becomes visible to the tensor cores
        tc_fence_before();
        __syncthreads();
        if (warp == 0) {
            tc_fence_after();
            const unsigned a0 = sStg + (unsigned)(st % WG_ST) * stage_bytes, b0 = a0 + p.abytes;
            const unsigned hi = sdesc_hi(128u);  // 8 rows (channels) to the next 8
#pragma unroll
            for (int ks = 0; ks < WG_VS / 16; ks++)  // K blocks of 8 voxels: 2,048 and 16 N bytes apart
                tc_mma_elect(tmem, dpair(sdesc_lo(a0 + (unsigned)ks * 4096u, 2048u), hi),
                             dpair(sdesc_lo(b0 + (unsigned)ks * (unsigned)p.N * 32u, (unsigned)p.N * 16u), hi), p.idesc,
                             (st > 0 || ks > 0) ? 1u : 0u);
            tc_commit_elect(sb + 8u * (unsigned)(st % WG_ST));
        }
        issued = st;
        // the buffer of stage st + 2 is the one of stage st - 1, whose MMAs
        // were issued one iteration ago
        if (st >= 1) {
            const int q = st - 1;
            ok = __syncthreads_and(mb_wait(sb + 8u * (unsigned)(q % WG_ST), (unsigned)((q / WG_ST) & 1), abort_flag, p.err,
                                           21));
            if (!ok) break;
        }
        if (st + 2 < nstage) load(st + 2);
        else asm volatile("cp.async.commit_group;\n" ::: "memory");
    }
    asm volatile("cp.async.wait_all;\n" ::: "memory");  // no copy outlives the CTA
    // the last stage's MMAs (every commit of a barrier before it completed in order)
    if (ok && nstage > 0) {
        const int sl = nstage - 1;
        ok = __all_sync(0xffffffffu, mb_wait(sb + 8u * (unsigned)(sl % WG_ST), (unsigned)((sl / WG_ST) & 1), abort_flag,
                                             p.err, 22));
        ok = __syncthreads_and(ok);
    }
    if (ok && nstage > 0) {
        tc_fence_after();
        const int r = 32 * warp + lane;
        const int s = r / p.C, c = r - s * p.C;
        const bool live = s < ntap && c < p.Cw;
        const unsigned lane_addr = (unsigned)(32 * warp) << 16;
        const bool v4 = (reinterpret_cast<uintptr_t>(p.dw) & 15) == 0;
        for (int n0 = 0; n0 < p.N; n0 += 16) {
            float v[16];
            __syncwarp();
            tc_ld16(tmem + lane_addr + (unsigned)n0, v);
            if (live) {
                float *d = p.dw + ((long long)(t0 + s) * p.Cw + c) * p.N + n0;
                if (v4) {
#pragma unroll
                    for (int j = 0; j < 16; j += 4) red_v4_f32(d + j, v[j], v[j + 1], v[j + 2], v[j + 3]);
                } else {
#pragma unroll
                    for (int j = 0; j < 16; j++) atomicAdd(d + j, v[j]);
                }
            }
        }
    }
    if (!ok && issued >= 0 && tid == 0)  // no MMA outlives the CTA: its last commit covers the earlier ones
        mb_wait(sb + 8u * (unsigned)(issued % WG_ST), (unsigned)((issued / WG_ST) & 1), abort_flag, p.err, 23, false);
    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(p.tmem_cols)
                     : "memory");
    }
}

}  // namespace

// z-taps in N for the thin layers, which are otherwise bound by the
// shared-memory reads of A: when N <= 32 and the resident weights fit beside
// two halo buffers of two-plane tiles.
static bool dzn_fits(int N, int K, int zt, int nbuf, unsigned *smem, unsigned *cols, unsigned *plane,
                     unsigned *halo, unsigned *off_h)
{
    const unsigned wbytes = 27u * (unsigned)N * (unsigned)K * 2u;
    *plane = plane_bytes(zt);
    *halo = (unsigned)(K / 8) * *plane;
    *off_h = (HDR + wbytes + 127u) & ~127u;
    *smem = ALIGN_SLACK + *off_h + (unsigned)nbuf * *halo;
    const unsigned acc = (unsigned)(zt * N);
    *cols = pow2_at_least((unsigned)nbuf * acc);
    return *smem <= TC_SMEM_MAX && zt * N <= 128;
}

bool conv3_tc_dzn(int N, int K)
{
    unsigned a, b, c, d, e;
    return N >= 16 && N <= 32 && (N % 16) == 0 && K >= 16 && (K % 16) == 0 && dzn_fits(N, K, 2, 2, &a, &b, &c, &d, &e);
}

int conv3_tc_plans(int N, int K, int D, TcPlan *out, int cap)
{
    if (N < 16 || N > 256 || (N % 16) || K < 16 || (K % 16) || cap < 1) return 0;
    int np = 0;
    if (conv3_tc_dzn(N, K)) {
        // the weights are packed for the dz-in-N MMA: only such plans apply
        static const int zd[] = {8, 4, 2};
        const int nbuf = 2;
        for (int zt : zd) {
            if (zt > 2 && zt > D) continue;
            unsigned smem, cols, plane, halo, off_h;
            if (!dzn_fits(N, K, zt, nbuf, &smem, &cols, &plane, &halo, &off_h)) continue;
            TcPlan &pl = out[np];
            pl.Zt = zt;
            pl.nbuf = nbuf;
            pl.nacc = nbuf;
            pl.wstages = 0;
            pl.dzn = 1;
            pl.plane = plane;
            pl.halo = halo;
            pl.off_w = HDR;
            pl.off_h = off_h;
            pl.wbytes = 27u * (unsigned)N * (unsigned)K * 2u;
            pl.smem = smem;
            pl.tmem_cols = cols;
            if (++np == cap) return np;
        }
        return np;
    }
    const unsigned wtap = (unsigned)N * (unsigned)K * 2u;
    static const int zts[] = {4, 2, 1};
    // resident weights first (even single-buffered: streaming the weights
    // costs more than the lost overlap); then a ring of 4, 3, 2 one-tap stages
    for (int stages = 0; stages <= MAX_WSTAGE; stages = stages ? stages - 1 : MAX_WSTAGE) {
        if (stages == 1) break;
        const unsigned wbytes = (stages ? (unsigned)stages : 27u) * wtap;
        for (int nbuf = 2; nbuf >= 1; nbuf--) {
            for (int zt : zts) {
                if (zt > 1 && zt > D) continue;
                const unsigned plane = plane_bytes(zt);
                const unsigned halo = (unsigned)(K / 8) * plane;
                const unsigned off_w = HDR;
                const unsigned off_h = (off_w + wbytes + 127u) & ~127u;
                const unsigned smem = ALIGN_SLACK + off_h + (unsigned)nbuf * halo;
                const int nacc = 2 * zt * N <= 512 ? 2 : 1;
                const unsigned cols = pow2_at_least((unsigned)(nacc * zt * N));
                if (smem > TC_SMEM_MAX || cols > 512) continue;
                TcPlan &pl = out[np];
                pl.Zt = zt;
                pl.nbuf = nbuf;
                pl.nacc = nacc;
                pl.wstages = stages;
                pl.dzn = 0;
                pl.plane = plane;
                pl.halo = halo;
                pl.off_w = off_w;
                pl.off_h = off_h;
                pl.wbytes = wbytes;
                pl.smem = smem;
                pl.tmem_cols = cols;
                if (++np == cap) return np;
            }
        }
    }
    return np;
}

bool conv3_tc_plan(int N, int K, int D, TcPlan *pl)
{
    return conv3_tc_plans(N, K, D, pl, 1) == 1;
}

using TcKernel = void (*)(const CUtensorMap, const CUtensorMap, const TcArgs);

// The instantiations: the usual tile shapes with compile-time operands, and
// one run-time variant per mode for the rest.
struct TcVariant {
    int dzn, zt, nks, n;
    TcKernel k;
};
#define TC_V(dz, zt, nks, n) {dz, zt, nks, n, k_conv3_tc<dz, zt, nks, n>}
#define TC_PLAIN(n) \
    TC_V(0, 4, 2, n), TC_V(0, 2, 2, n), TC_V(0, 1, 2, n), TC_V(0, 4, 4, n), TC_V(0, 2, 4, n), TC_V(0, 1, 4, n)
const TcVariant TC_VARIANTS[] = {TC_V(1, 8, 1, 16), TC_V(1, 4, 1, 16), TC_V(1, 4, 2, 16), TC_V(1, 4, 1, 32),
                                 TC_V(1, 4, 2, 32), TC_PLAIN(32),      TC_PLAIN(64),      TC_PLAIN(128),
                                 TC_V(1, 0, 0, 0),  TC_V(0, 0, 0, 0)};
#undef TC_PLAIN
#undef TC_V

TcKernel pick_kernel(const TcPlan &pl, int N, int K)
{
    const int nks = K >> 4, block = pl.dzn ? nks : (nks % 4 == 0 ? 4 : (nks % 2 == 0 ? 2 : 1));
    for (const TcVariant &v : TC_VARIANTS)
        if (v.dzn == pl.dzn && (!v.n || (v.zt == pl.Zt && v.nks == block && v.n == N))) return v.k;
    return nullptr;
}

// CTAs of a plan that fit on an SM, by shared memory and by TMEM.
static int ctas_by_smem(const TcPlan &pl) { return (int)(TC_SMEM_SM / (pl.smem + 1024u)); }
static int ctas_by_tmem(const TcPlan &pl) { return (int)(512u / pl.tmem_cols); }

// The rule's choice among the plain plans, by an estimate of the time of the SM
// with the most tiles in units of one z-plane's MMAs: every tile costs its
// planes plus what its start and end leave the tensor core idle, least with two
// CTAs on the SM (0.45), more with one and two halo buffers (0.6), most with one
// halo buffer (1.1), and 0.15 for streamed weights.  Measured (tile depth,
// buffers, weights): 64 -> 32 channels on 32 x 32^3 voxels 212 us with 2, 1,
// resident, 180 with 2, 1, streamed (two CTAs on an SM); 128 -> 64 on 32 x 16^3
// 85 with 1, 1, streamed, 71 with 2, 1, streamed, but on one 16^3 region 16
// against 22.  The dz-in-N plans keep their order: their depth decides the order
// of the sums.
static int choose_plan(const TcPlan *pl, int np, const TcConv &c)
{
    int best = 0;
    double least = 1e300;
    for (int k = 0; k < np; k++) {
        if (pl[k].dzn) return 0;
        const long long t = (long long)((c.W + 7) / 8) * ((c.H + 15) / 16) * ((c.D + pl[k].Zt - 1) / pl[k].Zt) * c.B;
        const int per_sm = std::max(1, std::min(2, std::min(ctas_by_smem(pl[k]), ctas_by_tmem(pl[k]))));
        const long long slots = (long long)device_sms() * per_sm;
        const double idle = per_sm > 1 ? 0.45 : (pl[k].nbuf > 1 ? 0.6 : 1.1);
        const double est = (double)(per_sm * ((t + slots - 1) / slots)) * (pl[k].Zt + idle + (pl[k].wstages ? 0.15 : 0.0));
        if (est < least * 0.999) {
            least = est;
            best = k;
        }
    }
    return best;
}

int conv3_tc(const TcConv &c, int *err, cudaStream_t s)
{
    const int K = c.C1 + c.C2, N = c.N;
    TcPlan plans[TC_MAX_PLANS];
    const int np = conv3_tc_plans(N, K, c.D, plans, TC_MAX_PLANS);
    if ((c.C1 % 8) || (c.C2 % 8) || (c.O1 % 16) || c.O1 > N || np < 1) return 0;
    const TcPlan pl = plans[c.plan >= 0 && c.plan < np ? c.plan : choose_plan(plans, np, c)];
    if ((reinterpret_cast<uintptr_t>(c.w) & 15) || (reinterpret_cast<uintptr_t>(c.in1) & 15) ||
        (c.C2 && (reinterpret_cast<uintptr_t>(c.in2) & 15)))
        return 0;
    // from here on the shape is supported: a failure is an error, not a fallback
    CUtensorMap m1, m2;
    const int zh = pl.Zt + 2;
    if (!make_map(&m1, c.in1, c.C1, c.B, c.D, c.H, c.W, zh)) return -1;
    if (c.C2 > 0) {
        if (!make_map(&m2, c.in2, c.C2, c.B, c.D, c.H, c.W, zh)) return -1;
    } else {
        m2 = m1;
    }
    static std::once_flag once;
    static cudaError_t attr_err = cudaSuccess;
    std::call_once(once, []() {
        for (const TcVariant &v : TC_VARIANTS) {
            cudaError_t e = cudaFuncSetAttribute(v.k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TC_SMEM_MAX);
            if (e != cudaSuccess) attr_err = e;
        }
    });
    if (attr_err != cudaSuccess) return -1;
    TcArgs a;
    a.w = c.w;
    a.bias = c.bias;
    a.out1 = c.out1;
    a.out2 = c.out2 ? c.out2 : c.out1;
    a.N = N;
    a.K = K;
    a.C1 = c.C1;
    a.O1 = c.O1;
    a.relu = c.relu;
    a.B = c.B; a.D = c.D; a.H = c.H; a.W = c.W;
    a.Zt = pl.Zt;
    a.nbuf = pl.nbuf;
    a.nacc = pl.nacc;
    a.wstages = pl.wstages;
    a.dzn = pl.dzn;
    a.acc_cols = (unsigned)(pl.Zt * N);
    a.tx = (c.W + 7) / 8;
    a.ty = (c.H + 15) / 16;
    a.tz = (c.D + pl.Zt - 1) / pl.Zt;
    a.ntiles = (long long)a.tx * a.ty * a.tz * c.B;
    a.wbytes = pl.wbytes;
    a.plane = pl.plane;
    a.halo = pl.halo;
    a.off_w = pl.off_w;
    a.off_h = pl.off_h;
    a.tx_bytes = (unsigned)(K / 8) * (unsigned)zh * ZSTRIDE + c.tx_extra;
    a.tmem_cols = pl.tmem_cols;
    a.err = err;
    const int per_sm_smem = ctas_by_smem(pl), per_sm_tmem = ctas_by_tmem(pl);
    int per_sm = per_sm_smem < per_sm_tmem ? per_sm_smem : per_sm_tmem;
    if (per_sm < 1) per_sm = 1;
    // never more CTAs on an SM than their TMEM allocations fit
    unsigned smem = pl.smem;
    if (per_sm_smem > per_sm_tmem && smem < TC_SMEM_SM / (unsigned)per_sm_tmem - 1024u)
        smem = TC_SMEM_SM / (unsigned)per_sm_tmem - 1024u;
    if (smem > TC_SMEM_MAX) smem = TC_SMEM_MAX;
    long long grid = (long long)device_sms() * per_sm;
    if (grid > a.ntiles) grid = a.ntiles;
    if (grid < 1) return 1;
    counted(pick_kernel(pl, N, K))<<<(unsigned)grid, TC_THREADS, smem, s>>>(m1, m2, a);
    return cudaGetLastError() == cudaSuccess ? 1 : -1;
}

bool up2_tc_ok(int N, int K, long long Vc)
{
    return N >= 8 && N % 8 == 0 && 8 * N <= 512 && K >= 16 && K % 16 == 0 && Vc % 128 == 0 &&
           UP_HDR + ALIGN_SLACK + (unsigned)K / 8u * 2048u + (unsigned)K * 16u * (unsigned)N <= TC_SMEM_MAX;
}

int up2_tc(const bf16 *in, const bf16 *w, const float *bias, bf16 *out, int B, int Dc, int K, int N, int *err,
           cudaStream_t s)
{
    const long long Vc = (long long)Dc * Dc * Dc;
    if (!up2_tc_ok(N, K, Vc) || (reinterpret_cast<uintptr_t>(in) & 15) || (reinterpret_cast<uintptr_t>(w) & 15) ||
        (reinterpret_cast<uintptr_t>(out) & 15))
        return 0;
    static std::once_flag once;
    static cudaError_t attr_err = cudaSuccess;
    std::call_once(once, []() {
        attr_err = cudaFuncSetAttribute(k_up2_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TC_SMEM_MAX);
    });
    if (attr_err != cudaSuccess) return -1;
    Up2Args a;
    a.in = in; a.w = w; a.bias = bias; a.out = out;
    a.K = K; a.N = N; a.Dc = Dc; a.Vc = Vc;
    a.ntiles = (long long)B * Vc / 128;
    a.abytes = (unsigned)K / 8u * 2048u;
    a.wbytes = (unsigned)K * 16u * (unsigned)N;  // 8 N rows x K x 2 bytes
    const unsigned ncols = 8u * (unsigned)N;
    a.nsplit = ncols > 256u ? 2u : 1u;
    a.ncols_split = ncols / a.nsplit;
    a.tmem_cols = pow2_at_least(ncols);
    a.idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((a.ncols_split >> 3) << 17) | ((128u >> 4) << 24);
    a.err = err;
    // at most as many CTAs per SM as their TMEM allocations fit: size the
    // shared-memory request so that no allocation has to wait
    const unsigned need = ALIGN_SLACK + UP_HDR + a.abytes + a.wbytes;
    const unsigned per_sm = 512u / a.tmem_cols;
    unsigned smem = TC_SMEM_SM / per_sm - 1024u;
    if (smem > TC_SMEM_MAX) smem = TC_SMEM_MAX;
    if (smem < need) smem = need;
    if (a.ntiles < 1) return 1;
    counted(k_up2_tc)<<<(unsigned)a.ntiles, 128, smem, s>>>(a);
    return cudaGetLastError() == cudaSuccess ? 1 : -1;
}

int wgrad3_tc(const bf16 *x1, int C1, const bf16 *x2, int C2, const bf16 *g, int Cg, int N, int Cw, float *dw, int B,
              int D, int *err, cudaStream_t s)
{
    const int C = C1 + C2;
    if (!(C == 16 || C == 32 || C == 64 || C == 128) || (C1 & 7) || N < 16 || N > 128 || (N & 15) || Cg < N ||
        (Cg & 7) || Cw > C || B < 1 || D < 1 || D > 1024)
        return 0;
    if ((reinterpret_cast<uintptr_t>(x1) & 15) || (C2 > 0 && (reinterpret_cast<uintptr_t>(x2) & 15)) ||
        (reinterpret_cast<uintptr_t>(g) & 15))
        return 0;
    static std::once_flag once;
    static cudaError_t attr_err = cudaSuccess;
    std::call_once(once, []() {
        attr_err = cudaFuncSetAttribute(k_wgrad_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TC_SMEM_MAX);
    });
    if (attr_err != cudaSuccess) return -1;
    WgTcArgs a;
    a.x1 = x1; a.x2 = C2 > 0 ? x2 : x1; a.C1 = C1; a.C = C;
    a.g = g; a.Cg = Cg; a.N = N; a.Cw = Cw; a.dw = dw; a.B = B; a.D = D;
    a.ntap = 128 / C;
    const int ntg = (27 + a.ntap - 1) / a.ntap;
    a.V = (long long)B * D * D * D;
    const long long target = std::max(1LL, 4LL * device_sms() / ntg);
    long long chunk = (a.V + target - 1) / target;
    chunk = std::max<long long>(WG_VS, (chunk + WG_VS - 1) / WG_VS * WG_VS);
    a.chunk = chunk;
    a.nchunk = (int)((a.V + chunk - 1) / chunk);
    a.abytes = 128u * WG_VS * 2u;
    a.bbytes = (unsigned)N * WG_VS * 2u;
    a.tmem_cols = pow2_at_least((unsigned)N);
    // BF16 x BF16 -> FP32, both operands MN-major (bits 15 and 16)
    a.idesc = (1u << 4) | (1u << 7) | (1u << 10) | (1u << 15) | (1u << 16) | (((unsigned)N >> 3) << 17) |
              ((128u >> 4) << 24);
    a.err = err;
    // at most as many CTAs per SM as their TMEM allocations fit
    const unsigned need = ALIGN_SLACK + WG_HDR + (unsigned)WG_ST * (a.abytes + a.bbytes);
    const unsigned per_sm = 512u / a.tmem_cols;
    unsigned smem = TC_SMEM_SM / per_sm - 1024u;
    if (smem > TC_SMEM_MAX) smem = TC_SMEM_MAX;
    if (smem < need) smem = need;
    if (smem > TC_SMEM_MAX) return 0;
    counted(k_wgrad_tc)<<<dim3((unsigned)a.nchunk, (unsigned)ntg), 128, smem, s>>>(a);
    return cudaGetLastError() == cudaSuccess ? 1 : -1;
}

}  // namespace gnb
