// unet.cu -- the supernova surrogate's 3D U-Net: BF16 inference and training
// kernels with FP32 accumulation (Sec. 3.3 of Hirashima et al., SC'25: a
// U-Net of 3D convolutions predicting the gas 0.1 Myr after a supernova,
// trained with an MSE loss and Adam at batch size 1).
//
// Architecture (a reading; the paper gives no layer list): levels with
// widths base, 2 base, 4 base, 8 base; two 3^3 convolutions (zero "same"
// padding, ReLU) per level; 2^3 max-pool down; 2^3 stride-2 transposed
// convolution up; skip tensor concatenated before the up-sampled tensor; 1^3
// linear head.  Activations are BF16 and blocked by 8 channels:
// [batch][channel / 8][z][y][x][channel % 8], so that 8 channels of one
// voxel are one 16-byte piece and a run of x voxels of one channel group is
// contiguous (the tensor-core convolution loads its halo rows by TMA); the
// network input is padded to 16 channels.
//
// Every convolution-shaped product is one implicit GEMM (rows = output
// voxels, columns = output channels, K = taps x input channels) on the
// tensor cores: BF16 operands staged in shared memory by cp.async (double
// buffered), mma.sync m16n8k16 with FP32 accumulators, bias/ReLU/BF16
// conversion fused into the epilogue.  Weight gradients are a second implicit
// GEMM (rows = input channels, K = voxels) split over voxel chunks.
#include <cuda_bf16.h>

#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <vector>

#include "common.cuh"
#include "conv_tc.cuh"
#include "../../include/galnb_testing.h"

typedef __nv_bfloat16 bf16;

namespace gnb {

enum { IG_CONV3 = 0, IG_CONV1 = 1, IG_UP2 = 2, IG_DOWN2 = 3 };

__device__ __constant__ signed char c_taps[27][3] = {
    {-1, -1, -1}, {-1, -1, 0}, {-1, -1, 1}, {-1, 0, -1}, {-1, 0, 0}, {-1, 0, 1}, {-1, 1, -1}, {-1, 1, 0}, {-1, 1, 1},
    {0, -1, -1},  {0, -1, 0},  {0, -1, 1},  {0, 0, -1},  {0, 0, 0},  {0, 0, 1},  {0, 1, -1},  {0, 1, 0},  {0, 1, 1},
    {1, -1, -1},  {1, -1, 0},  {1, -1, 1},  {1, 0, -1},  {1, 0, 0},  {1, 0, 1},  {1, 1, -1},  {1, 1, 0},  {1, 1, 1}};

struct IgArgs {
    int mode;
    const bf16 *in1, *in2;  // input channels [0, C1) from in1, [C1, C1 + C2) from in2
    int C1, C2;
    const bf16 *w;          // [taps][Npad][Kp], Kp = C1 + C2 rounded up to 16 (zeros beyond)
    const float *bias;      // [N] or null
    int N, Npad;
    bf16 *out1, *out2;      // channels [0, O1) -> out1, [O1, N) -> out2
    int O1;
    float *outf;            // FP32 output with N channels (instead of out1/out2)
    int relu;
    int B, D, H, W;         // grid of the GEMM rows
};

// Offset of element (voxel v = b * Vs + s, channel c) of a C-channel blocked
// tensor whose grid has Vs voxels per batch entry.
__device__ __forceinline__ long long blk(long long v, int c, int C, long long Vs)
{
    long long b = v / Vs, s = v - b * Vs;
    return ((b * (C >> 3) + (c >> 3)) * Vs + s) * 8 + (c & 7);
}

__device__ __forceinline__ void cp_async16(void *smem, const void *g, int bytes)
{
    unsigned s = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(s), "l"(g), "r"(bytes));
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N)); }

__device__ __forceinline__ void mma_bf16(float *d, const unsigned *a, const unsigned *b)
{
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};\n"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

// Source voxel of GEMM row r for tap t (or -1 when it lies in the zero padding).
__device__ __forceinline__ long long ig_src(const IgArgs &p, long long r, int t)
{
    long long x = r % p.W, q = r / p.W;
    long long y = q % p.H;
    q /= p.H;
    long long z = q % p.D, b = q / p.D;
    if (p.mode == IG_CONV3) {
        long long zz = z + c_taps[t][0], yy = y + c_taps[t][1], xx = x + c_taps[t][2];
        if (zz < 0 || zz >= p.D || yy < 0 || yy >= p.H || xx < 0 || xx >= p.W) return -1;
        return ((b * p.D + zz) * p.H + yy) * p.W + xx;
    }
    if (p.mode == IG_DOWN2) {  // gather from the grid twice as fine
        long long zz = 2 * z + ((t >> 2) & 1), yy = 2 * y + ((t >> 1) & 1), xx = 2 * x + (t & 1);
        return ((b * 2 * p.D + zz) * 2 * p.H + yy) * 2 * p.W + xx;
    }
    return r;  // IG_CONV1, IG_UP2: the row's own voxel
}

// Output voxel of GEMM row r (IG_UP2 scatters into the grid twice as fine).
__device__ __forceinline__ long long ig_dst(const IgArgs &p, long long r, int t)
{
    if (p.mode != IG_UP2) return r;
    long long x = r % p.W, q = r / p.W;
    long long y = q % p.H;
    q /= p.H;
    long long z = q % p.D, b = q / p.D;
    long long zz = 2 * z + ((t >> 2) & 1), yy = 2 * y + ((t >> 1) & 1), xx = 2 * x + (t & 1);
    return ((b * 2 * p.D + zz) * 2 * p.H + yy) * 2 * p.W + xx;
}

#define IG_M 64
#define IG_ST 4  // staged K steps
#define IG_CTAS 152  // CTAs below which a launch takes fewer output channels per CTA
// NB = number of 8-column blocks per CTA (N tile = 8 NB).  What bounds it is the
// latency of a K step (few CTAs at the coarse levels, 8 at 8^3): four steps are
// in flight, and a thread decodes its row once and steps tap and channel by
// counters (with 64-bit divisions in every step and two steps in flight the
// input gradient of the 128 -> 64 channel up-sampling of one 8^3 grid took 52 us,
// now 13).
template <int NB>
__global__ void __launch_bounds__(128) k_igemm(IgArgs p)
{
    constexpr int NT = 8 * NB;
    __shared__ __align__(16) bf16 sA[IG_ST][IG_M][16];
    __shared__ __align__(16) bf16 sB[IG_ST][NT][16];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, gid = lane >> 2, tig = lane & 3;
    const long long M = (long long)p.B * p.D * p.H * p.W;
    const long long row0 = (long long)blockIdx.x * IG_M;
    const int n0 = blockIdx.y * NT;
    const int K = p.C1 + p.C2;
    const int ntap = p.mode == IG_CONV3 ? 27 : (p.mode == IG_DOWN2 ? 8 : 1);
    const int tapz = p.mode == IG_UP2 ? (int)blockIdx.z : 0;
    const int kch = (K + 15) / 16;  // (a width of an odd multiple of 8 leaves the last step half empty)
    const int Kp = 16 * kch;
    const int nsteps = ntap * kch;
    const long long Vrow = (long long)p.D * p.H * p.W;
    const long long VsA = p.mode == IG_DOWN2 ? 8 * Vrow : Vrow;  // voxels per batch entry of the source grid
    const long long VsO = p.mode == IG_UP2 ? 8 * Vrow : Vrow;    // ... and of the output grid
    float acc[NB][4];
#pragma unroll
    for (int j = 0; j < NB; j++) acc[j][0] = acc[j][1] = acc[j][2] = acc[j][3] = 0.f;

    // the row this thread stages, and the next step to stage
    const int sr = tid >> 1, half = tid & 1;
    const bool row_in = row0 + sr < M;
    const long long gr0 = row_in ? row0 + sr : 0, b0 = gr0 / Vrow;
    const int sv0 = (int)(gr0 - b0 * Vrow);
    const int x = sv0 % p.W, y = sv0 / p.W % p.H, z = sv0 / p.W / p.H;
    int st_t = 0, st_c = 0, slot = 0;
    long long src_v = -1;  // source voxel within the batch entry (-1: zero padding)
    auto tap_voxel = [&](int t) -> long long {
        if (!row_in) return -1;
        if (p.mode == IG_CONV3) {
            const int zz = z + c_taps[t][0], yy = y + c_taps[t][1], xx = x + c_taps[t][2];
            if (zz < 0 || zz >= p.D || yy < 0 || yy >= p.H || xx < 0 || xx >= p.W) return -1;
            return ((long long)zz * p.H + yy) * p.W + xx;
        }
        if (p.mode == IG_DOWN2)  // gather from the grid twice as fine
            return ((long long)(2 * z + ((t >> 2) & 1)) * 2 * p.H + (2 * y + ((t >> 1) & 1))) * 2 * p.W + (2 * x + (t & 1));
        return sv0;  // IG_CONV1, IG_UP2: the row's own voxel
    };
    auto stage = [&]() {
        if (st_c == 0) src_v = tap_voxel(st_t);
        {   // A: 64 rows x 16 channels, one 16-byte piece per thread
            const int c = st_c + 8 * half;
            const bf16 *src = p.in1;
            const bool in = src_v >= 0 && c < K;
            if (in)
                src = c < p.C1 ? p.in1 + ((b0 * (p.C1 >> 3) + (c >> 3)) * VsA + src_v) * 8
                               : p.in2 + ((b0 * (p.C2 >> 3) + ((c - p.C1) >> 3)) * VsA + src_v) * 8;
            cp_async16(&sA[slot][sr][8 * half], src, in ? 16 : 0);
        }
        const int wt = p.mode == IG_UP2 ? tapz : st_t;
        for (int q = tid; q < NT * 2; q += 128) {  // B: NT rows x 16 k
            const int n = q >> 1;
            const bool in = (n0 + n) < p.Npad;
            const bf16 *src = in ? p.w + ((long long)wt * p.Npad + n0 + n) * Kp + st_c + 8 * half : p.w;
            cp_async16(&sB[slot][n][8 * half], src, in ? 16 : 0);
        }
        if ((st_c += 16) >= Kp) { st_c = 0; st_t++; }
        slot = slot + 1 == IG_ST ? 0 : slot + 1;
    };

    for (int s = 0; s < IG_ST - 1; s++) {
        if (s < nsteps) stage();
        cp_async_commit();
    }
    for (int s = 0; s < nsteps; s++) {
        const int buf = s % IG_ST;
        cp_async_wait<IG_ST - 2>();
        __syncthreads();  // step s has landed, and every warp is done with the slot staged next
        if (s + IG_ST - 1 < nsteps) stage();
        cp_async_commit();
        unsigned a[4];
        const int ra = 16 * warp + gid;
        a[0] = *reinterpret_cast<const unsigned *>(&sA[buf][ra][2 * tig]);
        a[1] = *reinterpret_cast<const unsigned *>(&sA[buf][ra + 8][2 * tig]);
        a[2] = *reinterpret_cast<const unsigned *>(&sA[buf][ra][2 * tig + 8]);
        a[3] = *reinterpret_cast<const unsigned *>(&sA[buf][ra + 8][2 * tig + 8]);
#pragma unroll
        for (int j = 0; j < NB; j++) {
            unsigned b[2];
            b[0] = *reinterpret_cast<const unsigned *>(&sB[buf][8 * j + gid][2 * tig]);
            b[1] = *reinterpret_cast<const unsigned *>(&sB[buf][8 * j + gid][2 * tig + 8]);
            mma_bf16(acc[j], a, b);
        }
    }
    // epilogue: bias, ReLU, BF16 (or FP32) store
#pragma unroll
    for (int h = 0; h < 2; h++) {
        long long gr = row0 + 16 * warp + gid + 8 * h;
        if (gr >= M) continue;
        long long ov = ig_dst(p, gr, tapz);
#pragma unroll
        for (int j = 0; j < NB; j++) {
            int col = n0 + 8 * j + 2 * tig;
            float v0 = acc[j][2 * h], v1 = acc[j][2 * h + 1];
            if (p.bias) {
                if (col < p.N) v0 += p.bias[col];
                if (col + 1 < p.N) v1 += p.bias[col + 1];
            }
            if (p.relu) { v0 = fmaxf(v0, 0.f); v1 = fmaxf(v1, 0.f); }
            if (p.outf) {
                if (col < p.N) p.outf[ov * p.N + col] = v0;
                if (col + 1 < p.N) p.outf[ov * p.N + col + 1] = v1;
            } else if (col + 1 < p.N || (col < p.N && (p.N & 1) == 0)) {
                __nv_bfloat162 pr = __floats2bfloat162_rn(v0, v1);
                if (col < p.O1) *reinterpret_cast<__nv_bfloat162 *>(p.out1 + blk(ov, col, p.O1, VsO)) = pr;
                else *reinterpret_cast<__nv_bfloat162 *>(p.out2 + blk(ov, col - p.O1, p.N - p.O1, VsO)) = pr;
            }
        }
    }
}

// Weight gradient dW[tap][ci][co] += sum_v X(v, tap)[ci] * G(v, tap)[co] over a
// chunk of GEMM rows v (split-K with FP32 atomics).  X is the forward input
// (concatenated from two tensors), G the output gradient.
struct WgArgs {
    int mode;
    const bf16 *x1, *x2;
    int C1, C2;
    const bf16 *g;
    int Cg;          // channels stored in g (>= N, multiple of 8)
    int N;           // output channels that exist in dW
    int Cw;          // input channels that exist in dW (<= C1 + C2; the padded network input has more)
    float *dw;       // [taps][Cw][N]
    int B, D, H, W;  // grid of the rows (coarse grid for IG_UP2)
    long long chunk; // rows per CTA
};

template <int NB>
__global__ void __launch_bounds__(128) k_wgrad(WgArgs p)
{
    constexpr int NT = 8 * NB;
    __shared__ __align__(16) bf16 sX[64][16 + 2];
    __shared__ __align__(16) bf16 sG[NT][16 + 2];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, gid = lane >> 2, tig = lane & 3;
    const long long M = (long long)p.B * p.D * p.H * p.W;
    const int t = blockIdx.z;
    const int ci0 = blockIdx.y * 64;
    const int Cin = p.C1 + p.C2;
    const long long r0 = (long long)blockIdx.x * p.chunk, r1 = min(M, r0 + p.chunk);
    IgArgs q;
    q.mode = p.mode; q.B = p.B; q.D = p.D; q.H = p.H; q.W = p.W;
    const long long VsX = (long long)p.D * p.H * p.W;                    // X lives on the row grid
    const long long VsG = p.mode == IG_UP2 ? 8 * VsX : VsX;              // G on the fine grid for IG_UP2
    float acc[NB][4];
#pragma unroll
    for (int j = 0; j < NB; j++) acc[j][0] = acc[j][1] = acc[j][2] = acc[j][3] = 0.f;
    for (long long rb = r0; rb < r1; rb += 16) {
        // X tile: 16 rows x 64 input channels, stored transposed [ci][row]
        for (int e = tid; e < 16 * 8; e += 128) {
            int rr = e >> 3, c8 = (e & 7) * 8;
            long long r = rb + rr;
            long long v = -1;
            if (r < r1) v = p.mode == IG_UP2 ? r : ig_src(q, r, t);
            int c = ci0 + c8;
            uint4 val = make_uint4(0, 0, 0, 0);
            if (v >= 0 && c < Cin)
                val = c < p.C1 ? *reinterpret_cast<const uint4 *>(p.x1 + blk(v, c, p.C1, VsX))
                               : *reinterpret_cast<const uint4 *>(p.x2 + blk(v, c - p.C1, p.C2, VsX));
            const bf16 *pv = reinterpret_cast<const bf16 *>(&val);
#pragma unroll
            for (int k = 0; k < 8; k++) sX[c8 + k][rr] = pv[k];
        }
        // G tile: 16 rows x NT output channels, stored transposed [co][row]
        for (int e = tid; e < 16 * NB; e += 128) {
            int rr = e / NB, c8 = (e % NB) * 8;
            long long r = rb + rr;
            uint4 val = make_uint4(0, 0, 0, 0);
            if (r < r1) {
                long long v = p.mode == IG_UP2 ? ig_dst(q, r, t) : r;
                if (c8 < p.Cg) val = *reinterpret_cast<const uint4 *>(p.g + blk(v, c8, p.Cg, VsG));
            }
            const bf16 *pv = reinterpret_cast<const bf16 *>(&val);
#pragma unroll
            for (int k = 0; k < 8; k++) sG[c8 + k][rr] = pv[k];
        }
        __syncthreads();
        unsigned a[4];
        const int ra = 16 * warp + gid;
        a[0] = *reinterpret_cast<const unsigned *>(&sX[ra][2 * tig]);
        a[1] = *reinterpret_cast<const unsigned *>(&sX[ra + 8][2 * tig]);
        a[2] = *reinterpret_cast<const unsigned *>(&sX[ra][2 * tig + 8]);
        a[3] = *reinterpret_cast<const unsigned *>(&sX[ra + 8][2 * tig + 8]);
#pragma unroll
        for (int j = 0; j < NB; j++) {
            unsigned b[2];
            b[0] = *reinterpret_cast<const unsigned *>(&sG[8 * j + gid][2 * tig]);
            b[1] = *reinterpret_cast<const unsigned *>(&sG[8 * j + gid][2 * tig + 8]);
            mma_bf16(acc[j], a, b);
        }
        __syncthreads();
    }
#pragma unroll
    for (int h = 0; h < 2; h++) {
        int ci = ci0 + 16 * warp + gid + 8 * h;
        if (ci >= p.Cw) continue;
#pragma unroll
        for (int j = 0; j < NB; j++) {
            int co = 8 * j + 2 * tig;
            float *d = p.dw + ((long long)t * p.Cw + ci) * p.N;
            if (co < p.N) atomicAdd(d + co, acc[j][2 * h]);
            if (co + 1 < p.N) atomicAdd(d + co + 1, acc[j][2 * h + 1]);
        }
    }
}

// ----------------------------------------------------------------- elementwise
// FP32 [V][cin] -> blocked BF16 with 16 channels (zeros beyond cin); Vs
// voxels per batch entry.
__global__ void __launch_bounds__(256) k_pack_input(const float *__restrict__ x, int cin, int B, int Vs,
                                                    bf16 *__restrict__ out)
{
    // one voxel per thread: its cin values, two 16-byte channel groups out
    const long long b = blockIdx.y + 65535LL * blockIdx.z;
    const int sv = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= B || sv >= Vs) return;
    const float *xv = x + (b * Vs + sv) * cin;
    float f[16];
#pragma unroll
    for (int c = 0; c < 16; c++) f[c] = c < cin ? xv[c] : 0.f;
#pragma unroll
    for (int g = 0; g < 2; g++) {
        uint4 o;
        unsigned *ou = reinterpret_cast<unsigned *>(&o);
#pragma unroll
        for (int q = 0; q < 4; q++) {
            __nv_bfloat162 h = __floats2bfloat162_rn(f[8 * g + 2 * q], f[8 * g + 2 * q + 1]);
            ou[q] = *reinterpret_cast<unsigned *>(&h);
        }
        *reinterpret_cast<uint4 *>(out + ((b * 2 + g) * Vs + sv) * 8) = o;
    }
}

// 1x1x1 head: FP32 out[v][n] = bias[n] + sum_k in(v)[k] w[n][k] for n < cout
// (<= 8) and k < C (<= 32, a multiple of 8); w is the packed BF16 [Npad][Kpad]
// forward weight.  One voxel per thread at a time; a block's outputs are staged
// in shared memory and leave as contiguous 16-byte stores.
constexpr int HEAD_T = 256, HEAD_R = 8;  // threads, and at most so many voxels per thread
template <int NO>
__global__ void __launch_bounds__(HEAD_T) k_head(const bf16 *__restrict__ in, int C, const bf16 *__restrict__ w,
                                                 int Kpad, const float *__restrict__ bias, int B, int Vs, int R,
                                                 float *__restrict__ out)
{
    // a block's voxels lie in one batch entry, given by the grid (a 64-bit
    // division a thread costs more than the products); weights [k][n]: one
    // input channel's are read together (16 bytes at a time instead of 128
    // single reads a voxel: 144 -> 122 us for 32 regions of 64^3, 65 at the copy
    // rate).  Eight voxels per thread pay once for staging the weights, and the
    // next voxel's loads are under way while one is summed (124 -> 93 us).
    constexpr int NP = (NO + 3) / 4 * 4;
    __shared__ __align__(16) float sw[32][NP], sbias[NP];
    __shared__ __align__(16) float so[2][HEAD_T * NO];
    const long long b = blockIdx.y + 65535LL * blockIdx.z;
    if (b >= B) return;
    const int v0 = blockIdx.x * HEAD_T * R, G = C >> 3;
    const bf16 *src = in + b * G * (long long)Vs * 8;
    uint4 u[4];
    auto load = [&](int sv) {
#pragma unroll
        for (int g = 0; g < 4; g++)
            if (g < G && sv < Vs) u[g] = *reinterpret_cast<const uint4 *>(src + ((long long)g * Vs + sv) * 8);
    };
    load(v0 + threadIdx.x);
    for (int i = threadIdx.x; i < 32 * NP; i += blockDim.x) {
        const int k = i / NP, n = i % NP;
        sw[k][n] = n < NO && k < C ? __bfloat162float(w[n * Kpad + k]) : 0.f;
    }
    if (threadIdx.x < NP) sbias[threadIdx.x] = threadIdx.x < NO && bias ? bias[threadIdx.x] : 0.f;
    __syncthreads();
#pragma unroll 1
    for (int it = 0; it < R && v0 + it * HEAD_T < Vs; it++) {
        const int vb = v0 + it * HEAD_T, sv = vb + threadIdx.x;
        float *st = so[it & 1];
        uint4 c[4];
#pragma unroll
        for (int g = 0; g < 4; g++) c[g] = u[g];
        if (it + 1 < R) load(sv + HEAD_T);
        if (sv < Vs) {
            float acc[NO];
#pragma unroll
            for (int n = 0; n < NO; n++) acc[n] = sbias[n];
#pragma unroll
            for (int g = 0; g < 4; g++) {
                if (g >= G) break;
                const __nv_bfloat162 *h = reinterpret_cast<const __nv_bfloat162 *>(&c[g]);
#pragma unroll
                for (int q = 0; q < 4; q++) {
                    const float2 f = __bfloat1622float2(h[q]);
                    float w0[NP], w1[NP];
#pragma unroll
                    for (int n = 0; n < NP; n += 4) {
                        *reinterpret_cast<float4 *>(w0 + n) = *reinterpret_cast<const float4 *>(&sw[8 * g + 2 * q][n]);
                        *reinterpret_cast<float4 *>(w1 + n) = *reinterpret_cast<const float4 *>(&sw[8 * g + 2 * q + 1][n]);
                    }
#pragma unroll
                    for (int n = 0; n < NO; n++) acc[n] += f.x * w0[n] + f.y * w1[n];
                }
            }
#pragma unroll
            for (int n = 0; n < NO; n++) st[threadIdx.x * NO + n] = acc[n];
        }
        __syncthreads();  // the other buffer's readers passed the barrier before
        const int nf = min(HEAD_T, Vs - vb) * NO;  // floats of this tile, contiguous
        float *dst = out + (b * Vs + vb) * NO;
        if ((reinterpret_cast<uintptr_t>(dst) & 15) == 0) {
            for (int i = threadIdx.x; i < nf / 4; i += HEAD_T)
                reinterpret_cast<float4 *>(dst)[i] = reinterpret_cast<const float4 *>(st)[i];
            for (int i = nf / 4 * 4 + threadIdx.x; i < nf; i += HEAD_T) dst[i] = st[i];
        } else {
            for (int i = threadIdx.x; i < nf; i += HEAD_T) dst[i] = st[i];
        }
    }
}

// Blocks of T threads over Vs voxels of each of B batch entries (y and z).
static dim3 batch_grid(long long Vs, int T, int B)
{
    return dim3((unsigned)((Vs + T - 1) / T), (unsigned)std::min(B, 65535), (unsigned)((B + 65534) / 65535));
}

__global__ void k_maxpool(const bf16 *__restrict__ in, bf16 *__restrict__ out, unsigned char *__restrict__ idx, int B,
                          int D, int H, int W, int C)
{
    // output grid (B, D, H, W); input grid twice as fine; q runs over the
    // blocked output's (b, channel group, voxel): 8 channels per thread, the
    // 2x2x2 inputs as 16-byte loads; the first maximum of the 8 taps wins
    long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const long long Vs = (long long)D * H * W;
    if (q >= (long long)B * (C >> 3) * Vs) return;
    long long s = q % Vs, bg = q / Vs;  // bg = b * C / 8 + channel group
    long long x = s % W, r = s / W, y = r % H, z = r / H;
    const bf16 *src = in + bg * 8 * Vs * 8;
    float best[8];
    unsigned bi[8];
#pragma unroll
    for (int t = 0; t < 8; t++) {
        long long zz = 2 * z + ((t >> 2) & 1), yy = 2 * y + ((t >> 1) & 1), xx = 2 * x + (t & 1);
        const uint4 u = *reinterpret_cast<const uint4 *>(src + ((zz * 2 * H + yy) * 2 * W + xx) * 8);
        const bf16 *h = reinterpret_cast<const bf16 *>(&u);
#pragma unroll
        for (int j = 0; j < 8; j++) {
            const float f = __bfloat162float(h[j]);
            if (t == 0 || f > best[j]) { best[j] = f; bi[j] = (unsigned)t; }
        }
    }
    uint4 o;
    bf16 *ob = reinterpret_cast<bf16 *>(&o);
    unsigned lo = 0, hi = 0;
#pragma unroll
    for (int j = 0; j < 8; j++) {
        ob[j] = __float2bfloat16_rn(best[j]);
        if (j < 4) lo |= bi[j] << (8 * j);
        else hi |= bi[j] << (8 * (j - 4));
    }
    *reinterpret_cast<uint4 *>(out + q * 8) = o;
    *reinterpret_cast<uint2 *>(idx + q * 8) = make_uint2(lo, hi);
}

// dIn (fine grid) = routed pool gradient + skip gradient; a thread takes one
// fine voxel's group of 8 channels (16-byte pieces)
__global__ void k_maxpool_bwd(const bf16 *__restrict__ dout, const unsigned char *__restrict__ idx,
                              const bf16 *__restrict__ dskip, bf16 *__restrict__ din, int B, int D, int H, int W, int C)
{
    // fine grid (B, 2D, 2H, 2W); q runs over the pieces of the blocked fine tensor
    const long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const long long Vc = (long long)D * H * W, Vf = 8 * Vc;
    if (q >= B * Vf * (C >> 3)) return;
    const long long bg = q / Vf;
    const int s = (int)(q - bg * Vf);
    const int x = s % (2 * W), r = s / (2 * W), y = r % (2 * H), z = r / (2 * H);
    const unsigned t = ((z & 1) << 2) | ((y & 1) << 1) | (x & 1);
    const long long cv = bg * Vc + ((long long)(z >> 1) * H + (y >> 1)) * W + (x >> 1);
    const uint2 iv = reinterpret_cast<const uint2 *>(idx)[cv];
    const uint4 dv = reinterpret_cast<const uint4 *>(dout)[cv];
    uint4 sv = make_uint4(0u, 0u, 0u, 0u), ov;
    if (dskip) sv = reinterpret_cast<const uint4 *>(dskip)[q];
    const bf16 *dp = reinterpret_cast<const bf16 *>(&dv), *sp = reinterpret_cast<const bf16 *>(&sv);
    bf16 *op = reinterpret_cast<bf16 *>(&ov);
#pragma unroll
    for (int j = 0; j < 8; j++) {
        const unsigned i = ((j < 4 ? iv.x : iv.y) >> (8 * (j & 3))) & 255u;
        float g = i == t ? __bfloat162float(dp[j]) : 0.f;
        if (dskip) g += __bfloat162float(sp[j]);
        op[j] = __float2bfloat16_rn(g);
    }
    reinterpret_cast<uint4 *>(din)[q] = ov;
}

// Blocked BF16 [B][C/8][V][8] -> FP32 [B][V][keep] (the first `keep` channels).
__global__ void k_unblock(const bf16 *__restrict__ in, int B, int C, long long V, int keep, float *__restrict__ out)
{
    long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= (long long)B * V * keep) return;
    int c = (int)(e % keep);
    long long bv = e / keep, b = bv / V, v = bv - b * V;
    out[e] = __bfloat162float(in[((b * (C >> 3) + (c >> 3)) * V + v) * 8 + (c & 7)]);
}

// MSE over (voxels, cout <= 8): loss partial sums in FP64 and dy = 2 (y - t) /
// count as BF16 with 16 channels (zeros beyond cout); a voxel per thread, one
// atomic per block (a fixed number of blocks).
__global__ void __launch_bounds__(256) k_mse(const float *__restrict__ y, const float *__restrict__ tgt, long long V,
                                             long long Vs, int cout, bf16 *__restrict__ dy, double *__restrict__ loss)
{
    __shared__ double sh[8];
    double l = 0.0;
    const float cnt = (float)(V * cout);
    for (long long v = (long long)blockIdx.x * blockDim.x + threadIdx.x; v < V; v += (long long)gridDim.x * blockDim.x) {
        uint4 o;
        bf16 *h = reinterpret_cast<bf16 *>(&o);
#pragma unroll
        for (int c = 0; c < 8; c++) {
            float g = 0.f;
            if (c < cout) {
                const float d = y[v * cout + c] - tgt[v * cout + c];
                l += (double)d * d;
                g = 2.f * d / cnt;
            }
            h[c] = __float2bfloat16_rn(g);
        }
        const long long b = v / Vs, s = v - b * Vs;
        uint4 *p = reinterpret_cast<uint4 *>(dy) + b * 2 * Vs + s;
        p[0] = o;
        p[Vs] = make_uint4(0u, 0u, 0u, 0u);  // channels 8 .. 15
    }
    l = warp_sum(l);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = l;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0;
        for (int q = 0; q < 8; q++) t += sh[q];
        atomicAdd(loss, t);
    }
}

// Column sums of a blocked BF16 tensor g (Vs voxels per batch entry, B entries,
// cg8 groups of 8 channels) into db[0 .. N), the bias gradient: block row y is a
// channel group, a thread adds up 16-byte pieces.  MASK: g is first set to
// zero where y <= 0 (the ReLU's backward) and written to dz, so the mask and
// the sums are one pass.
template <bool MASK>
__global__ void __launch_bounds__(256) k_colsum(const uint4 *__restrict__ g, const uint4 *__restrict__ y,
                                                uint4 *__restrict__ dz, int B, long long Vs, int cg8, int N,
                                                float *__restrict__ db)
{
    __shared__ float sh[8][8];
    const int cg = blockIdx.y, lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    float s[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    for (int b = 0; b < B; b++) {
        const long long p0 = ((long long)b * cg8 + cg) * Vs;
        for (long long v = p0 + (long long)blockIdx.x * blockDim.x + threadIdx.x; v < p0 + Vs;
             v += (long long)gridDim.x * blockDim.x) {
            const uint4 u = g[v];
            unsigned gi[4] = {u.x, u.y, u.z, u.w};
            if (MASK) {
                const uint4 m = y[v];
                const unsigned mi[4] = {m.x, m.y, m.z, m.w};
#pragma unroll
                for (int q = 0; q < 4; q++) {
                    const __nv_bfloat162 h = *reinterpret_cast<const __nv_bfloat162 *>(&mi[q]);
                    gi[q] = (__low2float(h) > 0.f ? gi[q] & 0xffffu : 0u) | (__high2float(h) > 0.f ? gi[q] & 0xffff0000u : 0u);
                }
                dz[v] = make_uint4(gi[0], gi[1], gi[2], gi[3]);
            }
#pragma unroll
            for (int q = 0; q < 4; q++) {
                const __nv_bfloat162 h = *reinterpret_cast<const __nv_bfloat162 *>(&gi[q]);
                s[2 * q] += __low2float(h);
                s[2 * q + 1] += __high2float(h);
            }
        }
    }
#pragma unroll
    for (int j = 0; j < 8; j++) {
        const float t = warp_sum(s[j]);
        if (lane == 0) sh[w][j] = t;
    }
    __syncthreads();
    if (threadIdx.x < 8 && cg * 8 + threadIdx.x < N) {
        float t = 0.f;
        for (int q = 0; q < 8; q++) t += sh[q][threadIdx.x];
        atomicAdd(&db[cg * 8 + threadIdx.x], t);
    }
}

// Weight gradient of the 1^3 head, dw[c][n] += sum_v x(v)[c] g(v)[n] with n <
// N <= 8: block row y is a group of 8 input channels, a thread keeps the 64
// sums of its voxels in registers.  (As a split-K mma.sync GEMM with 5 of 8
// columns used: 289 us for one 64^3 region, now 10.)
__global__ void __launch_bounds__(128) k_wgrad_head(const uint4 *__restrict__ x, int B, long long Vs, int cg8,
                                                    const uint4 *__restrict__ g, int gg8, int N, int Cw,
                                                    float *__restrict__ dw)
{
    __shared__ float sh[4][64];
    const int cg = blockIdx.y, lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    float acc[8][8];
#pragma unroll
    for (int c = 0; c < 8; c++)
#pragma unroll
        for (int n = 0; n < 8; n++) acc[c][n] = 0.f;
    for (int b = 0; b < B; b++) {
        const uint4 *px = x + ((long long)b * cg8 + cg) * Vs, *pg = g + (long long)b * gg8 * Vs;
        for (long long v = (long long)blockIdx.x * blockDim.x + threadIdx.x; v < Vs; v += (long long)gridDim.x * blockDim.x) {
            const uint4 ux = px[v], ug = pg[v];
            const __nv_bfloat162 *hx = reinterpret_cast<const __nv_bfloat162 *>(&ux);
            const __nv_bfloat162 *hg = reinterpret_cast<const __nv_bfloat162 *>(&ug);
            float fx[8], fg[8];
#pragma unroll
            for (int q = 0; q < 4; q++) {
                fx[2 * q] = __low2float(hx[q]);
                fx[2 * q + 1] = __high2float(hx[q]);
                fg[2 * q] = __low2float(hg[q]);
                fg[2 * q + 1] = __high2float(hg[q]);
            }
#pragma unroll
            for (int c = 0; c < 8; c++)
#pragma unroll
                for (int n = 0; n < 8; n++) acc[c][n] = __fmaf_rn(fx[c], fg[n], acc[c][n]);
        }
    }
#pragma unroll
    for (int c = 0; c < 8; c++)
#pragma unroll
        for (int n = 0; n < 8; n++) {
            const float t = warp_sum(acc[c][n]);
            if (lane == 0) sh[w][c * 8 + n] = t;
        }
    __syncthreads();
    if (threadIdx.x < 64) {
        const int c = cg * 8 + (threadIdx.x >> 3), n = threadIdx.x & 7;
        if (c < Cw && n < N)
            atomicAdd(&dw[c * N + n], sh[0][threadIdx.x] + sh[1][threadIdx.x] + sh[2][threadIdx.x] + sh[3][threadIdx.x]);
    }
}

// Adam (Kingma and Ba): m = b1 m + (1 - b1) g, v = b2 v + (1 - b2) g^2,
// p -= lr (m / (1 - b1^t)) / (sqrt(v / (1 - b2^t)) + eps).  The constants
// 1 - b1, 1 - b2 and the bias corrections 1 / (1 - b^t) come from the host in
// FP64, rounded once: formed in FP32, 1 - 0.999f and 1 - 0.999^t lose five
// significant digits to cancellation.
__global__ void k_adam(float *__restrict__ p, const float *__restrict__ g, float *__restrict__ m,
                       float *__restrict__ v, long long n, float lr, float b1, float ob1, float b2, float ob2,
                       float eps, float ic1, float ic2)
{
    long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    float gi = g[i];
    float mi = __fmaf_rn(b1, m[i], ob1 * gi);
    float vi = __fmaf_rn(b2, v[i], ob2 * (gi * gi));
    m[i] = mi;
    v[i] = vi;
    p[i] -= lr * (mi * ic1) / (sqrtf(vi * ic2) + eps);
}

// One packed BF16 copy of a layer's FP32 master weights [taps][cin][cout]:
// rows n and columns k of each tap (forward: n = output, k = input channel;
// input gradient: the other way round, the taps of a 3^3 convolution mirrored,
// t -> taps - 1 - t), zero beyond the layer's channels, stored as
//   PK_PLAIN [taps][N][K];
//   PK_TC    [taps][K / 8][N][8], the tensor-core layout (up: one matrix of
//            the 8 taps' rows, [K / 8][8 N][8]);
//   PK_DZN   [9 (ty, tx)][K / 8][3 N (z-taps 2, 1, 0)][8], see conv3_tc_dzn.
enum { PK_PLAIN = 0, PK_TC, PK_UP, PK_DZN };
struct PackDesc {
    const float *w;
    bf16 *dst;
    int taps, cin, cout, N, K, layout, dgrad, mirror;
    long long total;
};

// All copies of a network in one launch, a block row per copy (four kernels a
// layer, 67 launches of 3.3 us each, before).
__global__ void __launch_bounds__(256) k_pack_weights(const PackDesc *__restrict__ table)
{
    const PackDesc d = table[blockIdx.y];
    for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < d.total; e += (long long)gridDim.x * blockDim.x) {
        int k, n, t;
        if (d.layout == PK_PLAIN) {
            k = (int)(e % d.K);
            const int q = (int)(e / d.K);
            n = q % d.N;
            t = q / d.N;
        } else {
            const int rows = d.layout == PK_UP ? 8 * d.N : (d.layout == PK_DZN ? 3 * d.N : d.N);
            const int j = (int)(e & 7), q = (int)(e >> 3), row = q % rows, r = q / rows;
            k = 8 * (r % (d.K / 8)) + j;
            const int m = r / (d.K / 8);
            n = row % d.N;
            t = d.layout == PK_UP ? row / d.N : (d.layout == PK_DZN ? 9 * (2 - row / d.N) + m : m);
        }
        if (d.mirror) t = d.taps - 1 - t;
        const int ci = d.dgrad ? n : k, co = d.dgrad ? k : n;
        d.dst[e] = __float2bfloat16_rn(ci < d.cin && co < d.cout ? d.w[((long long)t * d.cin + ci) * d.cout + co] : 0.f);
    }
}

}  // namespace gnb

// =================================================================== host
using namespace gnb;

namespace {

enum { L_CONV3 = 0, L_UP2 = 1, L_CONV1 = 2 };

struct ULayer {
    mutable int plan_f = -1;    // tile plan of the tensor-core forward convolution (-1: the rule's choice)
    int kind, cin, cout, taps;
    long long woff, boff;       // offsets in the flat parameter array
    int Npad, Kpad, Nd, Kd;     // padded forward / input-gradient GEMM shapes
    bf16 *wf = nullptr, *wd = nullptr;
    bf16 *wtc = nullptr, *wdtc = nullptr;  // tensor-core layouts of wf / wd (3^3 and up-sampling layers)
};

int round_up(int a, int b) { return (a + b - 1) / b * b; }

}  // namespace

struct gnb_unet {
    int cin, cout, base, levels, grid;
    cudaStream_t s;
    std::vector<ULayer> L;
    long long nparam = 0;
    float *p = nullptr, *g = nullptr, *m = nullptr, *v = nullptr;
    int adam_t = 0;
    // activations for batch capacity bcap
    int bcap = 0;
    std::vector<bf16 *> act;     // per stored tensor
    std::vector<unsigned char *> pidx;
    bf16 *xin = nullptr;
    float *yout = nullptr, *tgt = nullptr;
    bf16 *dyb = nullptr;
    std::vector<bf16 *> tmp;     // backward scratch
    double *loss_d = nullptr;
    int *err_d = nullptr;        // device error word of the tcgen05 convolutions
    int conv_impl = GNB_CONV_AUTO;
    unsigned tx_extra = 0;       // wait-timeout test only
    void *pack_d = nullptr;      // PackDesc table of the packed weight copies
    int npack = 0;
    bool launch_failed = false;
    bool tuning = false;         // forward passes time every tile plan of each 3^3 layer (gnb_unet_autotune)
    int tuned_layers = 0;
    uint64_t gen = 0;            // of the buffers and kernels a captured forward pass has in it (unet_generation)
    std::string err;
};

namespace {

// A number that no network has had before: of a new network, of new activation
// buffers or of another choice of kernels.
void new_generation(gnb_unet *u)
{
    static std::atomic<uint64_t> last{0};
    u->gen = ++last;
}

void unet_free_acts(gnb_unet *u)
{
    new_generation(u);
    for (auto *a : u->act) if (a) cudaFree(a);
    for (auto *a : u->pidx) if (a) cudaFree(a);
    for (auto *a : u->tmp) if (a) cudaFree(a);
    u->act.clear(); u->pidx.clear(); u->tmp.clear();
    if (u->xin) cudaFree(u->xin);
    if (u->yout) cudaFree(u->yout);
    if (u->tgt) cudaFree(u->tgt);
    if (u->dyb) cudaFree(u->dyb);
    u->xin = nullptr; u->yout = nullptr; u->tgt = nullptr; u->dyb = nullptr;
    u->bcap = 0;
}

// Tensor slots (index into act): per level l: 4 l + {0: enc a, 1: enc b (skip), 2: pool out}
// decoder level l: base 4 * levels + 3 l + {0: up, 1: dec a, 2: dec b}
int S_ENCA(int l) { return 4 * l; }
int S_ENCB(int l) { return 4 * l + 1; }
int S_POOL(int l) { return 4 * l + 2; }
int S_UP(const gnb_unet *u, int l) { return 4 * u->levels + 3 * l; }
int S_DECA(const gnb_unet *u, int l) { return 4 * u->levels + 3 * l + 1; }
int S_DECB(const gnb_unet *u, int l) { return 4 * u->levels + 3 * l + 2; }

int width(const gnb_unet *u, int l) { return u->base << l; }
long long vox(const gnb_unet *u, int l, int B) { long long g = u->grid >> l; return (long long)B * g * g * g; }

int unet_alloc_acts(gnb_unet *u, int B)
{
    if (u->bcap >= B) return GNB_OK;
    unet_free_acts(u);
    int nslot = 4 * u->levels + 3 * u->levels;
    u->act.assign(nslot, nullptr);
    u->pidx.assign(u->levels, nullptr);
    auto al = [&](void **p, size_t bytes) { return cudaMalloc(p, bytes) == cudaSuccess; };
    bool ok = true;
    for (int l = 0; l < u->levels; l++) {
        size_t n = (size_t)vox(u, l, B) * width(u, l);
        ok &= al((void **)&u->act[S_ENCA(l)], n * 2) && al((void **)&u->act[S_ENCB(l)], n * 2);
        if (l + 1 < u->levels) {
            size_t np = (size_t)vox(u, l + 1, B) * width(u, l);
            ok &= al((void **)&u->act[S_POOL(l)], np * 2) && al((void **)&u->pidx[l], np);
        }
        if (l + 1 < u->levels) {
            ok &= al((void **)&u->act[S_UP(u, l)], n * 2) && al((void **)&u->act[S_DECA(u, l)], n * 2) &&
                  al((void **)&u->act[S_DECB(u, l)], n * 2);
        }
    }
    size_t v0 = (size_t)vox(u, 0, B);
    ok &= al((void **)&u->xin, v0 * 16 * 2) && al((void **)&u->yout, v0 * u->cout * 4) &&
          al((void **)&u->tgt, v0 * u->cout * 4) && al((void **)&u->dyb, v0 * 16 * 2);
    // backward scratch: 4 buffers of the largest level-0 tensor with 2 * base channels
    u->tmp.assign(4, nullptr);
    for (int k = 0; k < 4; k++) ok &= al((void **)&u->tmp[k], v0 * (size_t)(2 * u->base) * 2 + 256);
    if (!ok) {
        cudaGetLastError();
        unet_free_acts(u);
        return GNB_ENOMEM;
    }
    u->bcap = B;
    return GNB_OK;
}

template <int NB>
void launch_ig_nb(const IgArgs &a, int ntiles_n, int gz, cudaStream_t s)
{
    long long M = (long long)a.B * a.D * a.H * a.W;
    dim3 grid((unsigned)((M + IG_M - 1) / IG_M), ntiles_n, gz);
    counted(k_igemm<NB>)<<<grid, 128, 0, s>>>(a);
}

void launch_ig(const IgArgs &a, cudaStream_t s)
{
    // 8 NB output channels a CTA: all of them (at most 128), but while that
    // leaves most of the chip idle narrower ones, down to 16 (a training step of
    // one 64^3 region 1386 -> 1350 us, of two 32^3 regions 959 -> 924).
    const int gz = a.mode == IG_UP2 ? 8 : 1;
    const long long mt = ((long long)a.B * a.D * a.H * a.W + IG_M - 1) / IG_M * gz;
    int nb = 1;
    while (nb < 16 && 8 * nb < a.Npad) nb *= 2;
    while (nb > 2 && mt * ((a.Npad + 8 * nb - 1) / (8 * nb)) < IG_CTAS) nb /= 2;
    const int nt = (a.Npad + 8 * nb - 1) / (8 * nb);
    if (nb == 1) launch_ig_nb<1>(a, nt, gz, s);
    else if (nb == 2) launch_ig_nb<2>(a, nt, gz, s);
    else if (nb == 4) launch_ig_nb<4>(a, nt, gz, s);
    else if (nb == 8) launch_ig_nb<8>(a, nt, gz, s);
    else launch_ig_nb<16>(a, nt, gz, s);
}

template <int NB>
void launch_wg_nb(const WgArgs &a, int taps, cudaStream_t s)
{
    long long M = (long long)a.B * a.D * a.H * a.W;
    int cin = a.C1 + a.C2;
    dim3 grid((unsigned)((M + a.chunk - 1) / a.chunk), (cin + 63) / 64, taps);
    counted(k_wgrad<NB>)<<<grid, 128, 0, s>>>(a);
}

void launch_wg(WgArgs a, int taps, cudaStream_t s)
{
    long long M = (long long)a.B * a.D * a.H * a.W;
    long long want = M / 96 + 1;  // about 96 chunks per tap
    a.chunk = ((want + 15) / 16) * 16;
    if (a.chunk < 256) a.chunk = 256;
    int Np = round_up(a.N, 8);
    if (Np <= 8) launch_wg_nb<1>(a, taps, s);
    else if (Np <= 16) launch_wg_nb<2>(a, taps, s);
    else if (Np <= 32) launch_wg_nb<4>(a, taps, s);
    else if (Np <= 64) launch_wg_nb<8>(a, taps, s);
    else launch_wg_nb<16>(a, taps, s);
}

IgArgs ig_base(int mode, int B, int D, int H, int W)
{
    IgArgs a;
    memset(&a, 0, sizeof(a));
    a.mode = mode; a.B = B; a.D = D; a.H = H; a.W = W;
    return a;
}

// Table of the network's packed copies (made once, with the network).
int unet_pack_table(gnb_unet *u)
{
    std::vector<PackDesc> t;
    auto add = [&](const ULayer &l, bf16 *dst, bool dgrad, int layout) {
        if (!dst) return;
        PackDesc d;
        d.w = u->p + l.woff;
        d.dst = dst;
        d.taps = l.taps; d.cin = l.cin; d.cout = l.cout;
        d.N = dgrad ? l.Nd : l.Npad;
        d.K = dgrad ? l.Kd : l.Kpad;
        d.layout = layout;
        d.dgrad = dgrad;
        d.mirror = dgrad && l.kind == L_CONV3;
        d.total = (long long)l.taps * d.N * d.K;
        t.push_back(d);
    };
    auto tc = [](int N, int K) { return conv3_tc_dzn(N, K) ? PK_DZN : PK_TC; };
    for (auto &l : u->L) {
        add(l, l.wf, false, PK_PLAIN);
        add(l, l.wd, true, PK_PLAIN);
        add(l, l.wtc, false, l.kind == L_UP2 ? PK_UP : tc(l.Npad, l.Kpad));
        add(l, l.wdtc, true, tc(l.Nd, l.Kd));
    }
    u->npack = (int)t.size();
    if (cudaMalloc((void **)&u->pack_d, t.size() * sizeof(PackDesc)) != cudaSuccess) return GNB_ENOMEM;
    return cudaMemcpy(u->pack_d, t.data(), t.size() * sizeof(PackDesc), cudaMemcpyHostToDevice) == cudaSuccess ? GNB_OK
                                                                                                             : GNB_ECUDA;
}

int unet_pack(gnb_unet *u)
{
    counted(k_pack_weights)<<<dim3(64, (unsigned)u->npack), 256, 0, u->s>>>((const PackDesc *)u->pack_d);
    return cudaGetLastError() == cudaSuccess ? GNB_OK : GNB_ECUDA;
}

// layer index helpers (order of the flat parameter array)
int LI_ENCA(int l) { return 2 * l; }
int LI_ENCB(int l) { return 2 * l + 1; }
int LI_UP(const gnb_unet *u, int l) { return 2 * u->levels + 3 * (u->levels - 2 - l); }
int LI_DECA(const gnb_unet *u, int l) { return LI_UP(u, l) + 1; }
int LI_DECB(const gnb_unet *u, int l) { return LI_UP(u, l) + 2; }
int LI_HEAD(const gnb_unet *u) { return 2 * u->levels + 3 * (u->levels - 1); }

// The tcgen05 path for a 3^3 convolution: 1 launched, 0 not applicable, -1 error.
int conv3_try_tc(gnb_unet *u, const bf16 *wtc, int N, int B, int D, const bf16 *in1, int C1, const bf16 *in2, int C2,
                 const float *bias, bf16 *out1, int O1, bf16 *out2, int relu, int plan = -1)
{
    if (!wtc || u->conv_impl == GNB_CONV_MMA_SYNC) return 0;
    TcConv c;
    c.plan = plan;
    c.in1 = in1; c.in2 = in2 ? in2 : in1; c.C1 = C1; c.C2 = C2;
    c.w = wtc; c.bias = bias; c.N = N;
    c.out1 = out1; c.out2 = out2 ? out2 : out1; c.O1 = O1; c.relu = relu;
    c.B = B; c.D = D; c.H = D; c.W = D;
    c.tx_extra = u->tx_extra;
    u->tx_extra = 0;  // the wait-timeout test affects the first tensor-core launch only
    return conv3_tc(c, u->err_d, u->s);
}

// Tile autotuner of one tensor-core 3^3 layer: every supported plan (tile
// depth, halo buffers, resident or streamed weights) runs on the layer's real
// tensors, twice untimed and three times timed with CUDA events on the
// network's stream, and the fastest is kept for the layer's forward passes.
void tune_conv3(gnb_unet *u, const ULayer &ly, int B, int D, const bf16 *in1, int C1, const bf16 *in2, int C2,
                bf16 *out, int relu)
{
    TcPlan plans[TC_MAX_PLANS];
    const int np = conv3_tc_plans(ly.Npad, C1 + C2, D, plans, TC_MAX_PLANS);
    if (np < 2) return;
    cudaEvent_t e0, e1;
    if (cudaEventCreate(&e0) != cudaSuccess) return;
    if (cudaEventCreate(&e1) != cudaSuccess) { cudaEventDestroy(e0); return; }
    float best = 3.0e38f;
    int bi = -1;
    for (int k = 0; k < np; k++) {
        bool ok = true;
        for (int rep = 0; rep < 5 && ok; rep++) {
            if (rep == 2) cudaEventRecord(e0, u->s);
            ok = conv3_try_tc(u, ly.wtc, ly.Npad, B, D, in1, C1, in2, C2, u->p + ly.boff, out, ly.cout, nullptr, relu,
                              k) == 1;
        }
        cudaEventRecord(e1, u->s);
        float ms = 0.f;
        if (ok && cudaEventSynchronize(e1) == cudaSuccess && cudaEventElapsedTime(&ms, e0, e1) == cudaSuccess &&
            ms < best) {
            best = ms;
            bi = k;
        }
    }
    cudaGetLastError();
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    if (bi >= 0) ly.plan_f = bi;
    u->tuned_layers++;
}

void conv_fwd(gnb_unet *u, const ULayer &ly, int mode, int B, int D, const bf16 *in1, int C1, const bf16 *in2, int C2,
              bf16 *out, float *outf, int relu)
{
    if (mode == IG_CONV3 && !outf) {
        if (u->tuning && ly.wtc && u->conv_impl != GNB_CONV_MMA_SYNC) tune_conv3(u, ly, B, D, in1, C1, in2, C2, out, relu);
        int rc = conv3_try_tc(u, ly.wtc, ly.Npad, B, D, in1, C1, in2, C2, u->p + ly.boff, out, ly.cout, nullptr,
                              relu, ly.plan_f);
        if (rc != 0) { if (rc < 0) u->launch_failed = true; return; }
    }
    if (mode == IG_UP2 && !outf && !in2 && !relu && ly.wtc && C1 == ly.Kpad && ly.cout == ly.Npad &&
        u->conv_impl != GNB_CONV_MMA_SYNC) {
        int rc = up2_tc(in1, ly.wtc, u->p + ly.boff, out, B, D, C1, ly.Npad, u->err_d, u->s);
        if (rc != 0) { if (rc < 0) u->launch_failed = true; return; }
    }
    if (mode == IG_CONV1 && outf && !in2 && ly.Npad <= 8 && C1 % 8 == 0 && C1 <= 32 && ly.Kpad <= 32) {
        const int Vs = D * D * D;
        using Head = void (*)(const bf16 *, int, const bf16 *, int, const float *, int, int, int, float *);
        static const Head heads[8] = {k_head<1>, k_head<2>, k_head<3>, k_head<4>, k_head<5>, k_head<6>, k_head<7>, k_head<8>};
        // one voxel per thread while the blocks would not fill the chip (1216
        // of them), then up to HEAD_R
        const int R = (int)std::max(1LL, std::min<long long>(HEAD_R, (long long)B * Vs / (1216LL * HEAD_T)));
        counted(heads[ly.cout - 1])<<<batch_grid(Vs, HEAD_T * R, B), HEAD_T, 0, u->s>>>(in1, C1, ly.wf, ly.Kpad, u->p + ly.boff,
                                                                                       B, Vs, R, outf);
        return;
    }
    IgArgs a = ig_base(mode, B, D, D, D);
    a.in1 = in1; a.in2 = in2 ? in2 : in1; a.C1 = C1; a.C2 = C2;
    a.w = ly.wf; a.bias = u->p + ly.boff; a.N = ly.cout; a.Npad = ly.Npad;
    a.out1 = out; a.out2 = out; a.O1 = ly.cout; a.outf = outf; a.relu = relu;
    launch_ig(a, u->s);
}

// input gradient of a layer: dx (split in two when the input was a concatenation)
void conv_dgrad(gnb_unet *u, const ULayer &ly, int mode, int B, int D, const bf16 *dz, int Cz, bf16 *dx1, int O1,
                bf16 *dx2)
{
    if (mode == IG_CONV3 && Cz == ly.Kd) {
        int rc = conv3_try_tc(u, ly.wdtc, ly.Nd, B, D, dz, Cz, nullptr, 0, nullptr, dx1, O1, dx2, 0);
        if (rc != 0) { if (rc < 0) u->launch_failed = true; return; }
    }
    IgArgs a = ig_base(mode, B, D, D, D);
    a.in1 = dz; a.in2 = dz; a.C1 = Cz; a.C2 = 0;
    a.w = ly.wd; a.bias = nullptr; a.N = ly.cin; a.Npad = ly.Nd;
    a.out1 = dx1; a.out2 = dx2 ? dx2 : dx1; a.O1 = O1; a.outf = nullptr; a.relu = 0;
    launch_ig(a, u->s);
}

void conv_wgrad(gnb_unet *u, const ULayer &ly, int mode, int B, int D, const bf16 *x1, int C1, const bf16 *x2, int C2,
                const bf16 *g, int Cg)
{
    WgArgs a;
    memset(&a, 0, sizeof(a));
    a.mode = mode; a.x1 = x1; a.x2 = x2 ? x2 : x1; a.C1 = C1; a.C2 = C2; a.g = g; a.Cg = Cg; a.N = ly.cout;
    a.Cw = ly.cin;
    a.dw = u->g + ly.woff; a.B = B; a.D = D; a.H = D; a.W = D;
    // 3^3 layers on the tensor cores where the shape allows (tcgen05 GEMM
    // over (tap, channel) rows); the mma.sync GEMM otherwise
    int tc = 0;
    if (mode == IG_CONV3 && u->conv_impl == GNB_CONV_AUTO) {
        tc = wgrad3_tc(x1, C1, x2, x2 ? C2 : 0, g, Cg, ly.cout, ly.cin, a.dw, B, D, u->err_d, u->s);
        if (tc < 0) u->launch_failed = true;
    }
    if (mode == IG_CONV1 && !x2 && ly.cout <= 8 && u->conv_impl == GNB_CONV_AUTO) {
        const long long Vh = (long long)D * D * D;
        counted(k_wgrad_head)<<<dim3((unsigned)std::max(1LL, std::min((Vh + 511) / 512, 304LL)), (unsigned)(C1 / 8)), 128, 0,
                               u->s>>>(reinterpret_cast<const uint4 *>(x1), B, Vh, C1 / 8,
                                       reinterpret_cast<const uint4 *>(g), Cg / 8, ly.cout, ly.cin, a.dw);
        tc = 1;
    }
    if (tc == 0) launch_wg(a, ly.taps, u->s);
}

// Bias gradient of a layer: column sums of its output gradient g; with y (the
// layer's stored output) g is masked by the ReLU first and written to dz.
void conv_bgrad(gnb_unet *u, const ULayer &ly, int B, long long Vs, const bf16 *g, int Cg, const bf16 *y = nullptr,
                bf16 *dz = nullptr)
{
    const int cgs = y ? Cg / 8 : (ly.cout + 7) / 8;  // every group is masked; else those with real columns
    const int nblk = (int)std::max(1LL, std::min((Vs + 1023) / 1024, 608LL / cgs));
    const dim3 grid((unsigned)nblk, (unsigned)cgs);
    const uint4 *g4 = reinterpret_cast<const uint4 *>(g);
    if (y)
        counted(k_colsum<true>)<<<grid, 256, 0, u->s>>>(g4, reinterpret_cast<const uint4 *>(y), reinterpret_cast<uint4 *>(dz),
                                                        B, Vs, Cg / 8, ly.cout, u->g + ly.boff);
    else
        counted(k_colsum<false>)<<<grid, 256, 0, u->s>>>(g4, nullptr, nullptr, B, Vs, Cg / 8, ly.cout, u->g + ly.boff);
}

// Forward pass of B regions from the blocked BF16 input xin to the FP32
// output yout (defaults: the network's own buffers).
int unet_forward(gnb_unet *u, int B, const bf16 *xin = nullptr, float *yout = nullptr)
{
    int G = u->grid;
    const bf16 *h = xin ? xin : u->xin;
    int ch = 16;
    for (int l = 0; l < u->levels; l++) {
        int D = G >> l, w = width(u, l);
        conv_fwd(u, u->L[LI_ENCA(l)], IG_CONV3, B, D, h, ch, nullptr, 0, u->act[S_ENCA(l)], nullptr, 1);
        conv_fwd(u, u->L[LI_ENCB(l)], IG_CONV3, B, D, u->act[S_ENCA(l)], w, nullptr, 0, u->act[S_ENCB(l)], nullptr, 1);
        if (l + 1 < u->levels) {
            long long n = vox(u, l + 1, B) * w;
            counted(k_maxpool)<<<(unsigned)((n / 8 + 255) / 256), 256, 0, u->s>>>(u->act[S_ENCB(l)], u->act[S_POOL(l)],
                                                                                 u->pidx[l], B, D / 2, D / 2, D / 2, w);
            h = u->act[S_POOL(l)];
        } else {
            h = u->act[S_ENCB(l)];
        }
        ch = w;
    }
    for (int l = u->levels - 2; l >= 0; l--) {
        int D = G >> l, w = width(u, l);
        // up-sampling GEMM rows live on the coarse grid
        conv_fwd(u, u->L[LI_UP(u, l)], IG_UP2, B, D / 2, h, 2 * w, nullptr, 0, u->act[S_UP(u, l)], nullptr, 0);
        conv_fwd(u, u->L[LI_DECA(u, l)], IG_CONV3, B, D, u->act[S_ENCB(l)], w, u->act[S_UP(u, l)], w,
                 u->act[S_DECA(u, l)], nullptr, 1);
        conv_fwd(u, u->L[LI_DECB(u, l)], IG_CONV3, B, D, u->act[S_DECA(u, l)], w, nullptr, 0, u->act[S_DECB(u, l)],
                 nullptr, 1);
        h = u->act[S_DECB(u, l)];
    }
    conv_fwd(u, u->L[LI_HEAD(u)], IG_CONV1, B, G, h, u->base, nullptr, 0, nullptr, yout ? yout : u->yout, 0);
    return cudaGetLastError() == cudaSuccess && !u->launch_failed ? GNB_OK : GNB_ECUDA;
}

// Backward through the network for dy in u->dyb (16 channels); gradients
// accumulate into u->g (zeroed by the caller).
int unet_backward(gnb_unet *u, int B)
{
    int G = u->grid, b0 = u->base;
    cudaStream_t s = u->s;
    bf16 *T0 = u->tmp[0], *T1 = u->tmp[1], *T2 = u->tmp[2], *T3 = u->tmp[3];
    auto relu_mask = [&](const ULayer &ly, int D, const bf16 *dy, const bf16 *y, bf16 *dz) {
        conv_bgrad(u, ly, B, (long long)D * D * D, dy, ly.cout, y, dz);
    };
    // head
    const ULayer &hd = u->L[LI_HEAD(u)];
    const bf16 *top = u->act[S_DECB(u, 0)];
    conv_wgrad(u, hd, IG_CONV1, B, G, top, b0, nullptr, 0, u->dyb, 16);
    conv_bgrad(u, hd, B, (long long)G * G * G, u->dyb, 16);
    conv_dgrad(u, hd, IG_CONV1, B, G, u->dyb, 16, T0, b0, nullptr);  // T0: d(dec0b.out)
    // decoder levels 0 .. levels-2; skip gradients stay in the ENC slots' spare: use T-buffers per level
    // dskip[l] is stored in place of the decoder's "up" activation gradient area: allocate per level below
    std::vector<bf16 *> dskip(u->levels, nullptr);
    bf16 *dcur = T0;  // gradient of the current decoder output
    for (int l = 0; l + 1 < u->levels; l++) {
        int D = G >> l, w = width(u, l);
        // the level-l tensors are at most as large as level 0 with 2 * base channels
        relu_mask(u->L[LI_DECB(u, l)], D, dcur, u->act[S_DECB(u, l)], T1);
        conv_wgrad(u, u->L[LI_DECB(u, l)], IG_CONV3, B, D, u->act[S_DECA(u, l)], w, nullptr, 0, T1, w);
        conv_dgrad(u, u->L[LI_DECB(u, l)], IG_CONV3, B, D, T1, w, T2, w, nullptr);
        relu_mask(u->L[LI_DECA(u, l)], D, T2, u->act[S_DECA(u, l)], T1);
        conv_wgrad(u, u->L[LI_DECA(u, l)], IG_CONV3, B, D, u->act[S_ENCB(l)], w, u->act[S_UP(u, l)], w, T1, w);
        // dskip -> the level's dec-a slot (its forward value is no longer needed), dup -> T2
        dskip[l] = u->act[S_DECA(u, l)];
        conv_dgrad(u, u->L[LI_DECA(u, l)], IG_CONV3, B, D, T1, w, dskip[l], w, T2);
        // up-conv: weight gradient (rows on the coarse grid), input gradient by gather
        int Dc = D / 2, wc = 2 * w;
        conv_wgrad(u, u->L[LI_UP(u, l)], IG_UP2, B, Dc, l + 2 < u->levels ? u->act[S_DECB(u, l + 1)]
                                                                          : u->act[S_ENCB(u->levels - 1)],
                   wc, nullptr, 0, T2, w);
        conv_bgrad(u, u->L[LI_UP(u, l)], B, (long long)D * D * D, T2, w);
        conv_dgrad(u, u->L[LI_UP(u, l)], IG_DOWN2, B, Dc, T2, w, T3, wc, nullptr);
        std::swap(T0, T3);
        dcur = T0;  // gradient of the level-(l+1) decoder output (or the bottleneck)
    }
    // encoder, bottleneck first
    for (int l = u->levels - 1; l >= 0; l--) {
        int D = G >> l, w = width(u, l);
        long long n = vox(u, l, B) * w;
        if (l + 1 < u->levels) {
            // dcur is the gradient of pool(l) output; route it and add the skip gradient
            counted(k_maxpool_bwd)<<<(unsigned)((n / 8 + 255) / 256), 256, 0, s>>>(dcur, u->pidx[l], dskip[l], T3, B,
                                                                             D / 2, D / 2, D / 2, w);
            std::swap(T0, T3);
            dcur = T0;
        }
        relu_mask(u->L[LI_ENCB(l)], D, dcur, u->act[S_ENCB(l)], T1);
        conv_wgrad(u, u->L[LI_ENCB(l)], IG_CONV3, B, D, u->act[S_ENCA(l)], w, nullptr, 0, T1, w);
        conv_dgrad(u, u->L[LI_ENCB(l)], IG_CONV3, B, D, T1, w, T2, w, nullptr);
        relu_mask(u->L[LI_ENCA(l)], D, T2, u->act[S_ENCA(l)], T1);
        const bf16 *xin = l == 0 ? u->xin : u->act[S_POOL(l - 1)];
        int cin = l == 0 ? 16 : width(u, l - 1);
        conv_wgrad(u, u->L[LI_ENCA(l)], IG_CONV3, B, D, xin, cin, nullptr, 0, T1, w);
        if (l > 0) {
            conv_dgrad(u, u->L[LI_ENCA(l)], IG_CONV3, B, D, T1, w, T3, cin, nullptr);
            std::swap(T0, T3);
            dcur = T0;
        }
    }
    return cudaGetLastError() == cudaSuccess && !u->launch_failed ? GNB_OK : GNB_ECUDA;
}

// Synchronise and collect errors: launch failures, CUDA errors and the
// tcgen05 convolutions' device error word (a bounded wait that ran out).
int unet_check(gnb_unet *u, int rc)
{
    u->launch_failed = false;
    if (cudaStreamSynchronize(u->s) != cudaSuccess || cudaGetLastError() != cudaSuccess) return GNB_ECUDA;
    int e = 0;
    if (u->err_d) {
        if (cudaMemcpy(&e, u->err_d, sizeof(int), cudaMemcpyDeviceToHost) != cudaSuccess) return GNB_ECUDA;
        if (e != 0) {
            cudaMemsetAsync(u->err_d, 0, sizeof(int), u->s);
            cudaStreamSynchronize(u->s);
            return GNB_ETIMEOUT;
        }
    }
    return rc;
}

}  // namespace

namespace gnb {
// Hooks for the batched surrogate step: make room for `batch` regions and
// expose the blocked BF16 input [batch][2][grid^3][8] and the FP32 output
// [batch][grid^3][cout]; unet_run launches the forward pass of `batch`
// regions on `stream` without synchronising (so it can be captured in a CUDA
// graph), from xin to yout (null: those buffers' starts).
int unet_prepare(gnb_unet *u, int batch, bf16 **xin, float **yout, int *grid, int *cout)
{
    int rc = unet_alloc_acts(u, batch);
    if (rc != GNB_OK) return rc;
    *xin = u->xin;
    *yout = u->yout;
    *grid = u->grid;
    *cout = u->cout;
    return GNB_OK;
}

uint64_t unet_generation(const gnb_unet *u) { return u->gen; }

int unet_poll_error(gnb_unet *u)
{
    int e = 0;
    if (!u || !u->err_d || cudaMemcpy(&e, u->err_d, sizeof(int), cudaMemcpyDeviceToHost) != cudaSuccess) return GNB_OK;
    if (e == 0) return GNB_OK;
    cudaMemsetAsync(u->err_d, 0, sizeof(int), u->s);
    return GNB_ETIMEOUT;
}

int unet_run(gnb_unet *u, int batch, cudaStream_t stream, const bf16 *xin, float *yout)
{
    cudaStream_t keep = u->s;
    u->s = stream;
    int rc = unet_forward(u, batch, xin, yout);
    u->s = keep;
    return rc;
}
}  // namespace gnb

extern "C" {

int gnb_unet_create(gnb_unet **out, int cin, int cout, int base, int levels, int grid, void *stream)
{
    if (!out) return GNB_EINVAL;
    *out = nullptr;
    if (cin < 1 || cin > 16 || cout < 1 || cout > 8 || base < 8 || base > 32 || (base % 8) || levels < 2 ||
        levels > 5 || grid < 8 || (grid % (1 << (levels - 1))) || ((grid >> (levels - 1)) < 2))
        return GNB_EINVAL;
    gnb_unet *u = new (std::nothrow) gnb_unet();
    if (!u) return GNB_ENOMEM;
    u->cin = cin; u->cout = cout; u->base = base; u->levels = levels; u->grid = grid;
    u->s = (cudaStream_t)stream;
    new_generation(u);
    // layers in the order of the flat parameter array
    auto add = [&](int kind, int ci, int co) {
        ULayer l;
        l.kind = kind; l.cin = ci; l.cout = co;
        l.taps = kind == L_CONV3 ? 27 : (kind == L_UP2 ? 8 : 1);
        l.woff = u->nparam;
        u->nparam += (long long)l.taps * ci * co;
        l.boff = u->nparam;
        u->nparam += co;
        l.Kpad = round_up(ci, 16);
        l.Npad = round_up(co, 8);
        l.Nd = round_up(ci, 8);
        l.Kd = round_up(co, 16);
        u->L.push_back(l);
    };
    int c = 16;  // the network input is padded to 16 channels
    for (int l = 0; l < levels; l++) {
        add(L_CONV3, l == 0 ? cin : c, base << l);
        add(L_CONV3, base << l, base << l);
        c = base << l;
    }
    for (int l = levels - 2; l >= 0; l--) {
        add(L_UP2, base << (l + 1), base << l);
        add(L_CONV3, 2 * (base << l), base << l);
        add(L_CONV3, base << l, base << l);
    }
    add(L_CONV1, base, cout);
    // the first layer's input has 16 (padded) channels in the GEMM
    u->L[0].Kpad = 16;
    u->L[0].Nd = 16;
    bool ok = cudaMalloc((void **)&u->p, u->nparam * 4) == cudaSuccess &&
              cudaMalloc((void **)&u->g, u->nparam * 4) == cudaSuccess &&
              cudaMalloc((void **)&u->m, u->nparam * 4) == cudaSuccess &&
              cudaMalloc((void **)&u->v, u->nparam * 4) == cudaSuccess &&
              cudaMalloc((void **)&u->loss_d, 16) == cudaSuccess &&
              cudaMalloc((void **)&u->err_d, sizeof(int)) == cudaSuccess;
    for (auto &l : u->L) {
        ok = ok && cudaMalloc((void **)&l.wf, (size_t)l.taps * l.Npad * l.Kpad * 2) == cudaSuccess &&
             cudaMalloc((void **)&l.wd, (size_t)l.taps * l.Nd * l.Kd * 2) == cudaSuccess;
        TcPlan pl;
        if (ok && l.kind == L_CONV3 && conv3_tc_plan(l.Npad, l.Kpad, grid, &pl))
            ok = cudaMalloc((void **)&l.wtc, (size_t)l.taps * l.Npad * l.Kpad * 2) == cudaSuccess;
        if (ok && l.kind == L_UP2 && l.cin == l.Kpad && up2_tc_ok(l.Npad, l.Kpad, 128))
            ok = cudaMalloc((void **)&l.wtc, (size_t)l.taps * l.Npad * l.Kpad * 2) == cudaSuccess;
        if (ok && l.kind == L_CONV3 && conv3_tc_plan(l.Nd, l.Kd, grid, &pl))
            ok = cudaMalloc((void **)&l.wdtc, (size_t)l.taps * l.Nd * l.Kd * 2) == cudaSuccess;
    }
    if (!ok || unet_pack_table(u) != GNB_OK) {
        cudaGetLastError();
        gnb_unet_destroy(u);
        return GNB_ENOMEM;
    }
    cudaMemsetAsync(u->p, 0, u->nparam * 4, u->s);
    cudaMemsetAsync(u->g, 0, u->nparam * 4, u->s);
    cudaMemsetAsync(u->m, 0, u->nparam * 4, u->s);
    cudaMemsetAsync(u->v, 0, u->nparam * 4, u->s);
    cudaMemsetAsync(u->err_d, 0, sizeof(int), u->s);
    *out = u;
    return unet_check(u, unet_pack(u));
}

void gnb_unet_destroy(gnb_unet *u)
{
    if (!u) return;
    cudaStreamSynchronize(u->s);
    unet_free_acts(u);
    for (auto &l : u->L) {
        if (l.wf) cudaFree(l.wf);
        if (l.wd) cudaFree(l.wd);
        if (l.wtc) cudaFree(l.wtc);
        if (l.wdtc) cudaFree(l.wdtc);
    }
    float *a[] = {u->p, u->g, u->m, u->v};
    for (float *q : a) if (q) cudaFree(q);
    if (u->loss_d) cudaFree(u->loss_d);
    if (u->err_d) cudaFree(u->err_d);
    if (u->pack_d) cudaFree(u->pack_d);
    delete u;
}

int64_t gnb_unet_num_params(const gnb_unet *u) { return u ? u->nparam : -1; }

int gnb_unet_test_wait_timeout(gnb_unet *u)
{
    if (!u || u->conv_impl == GNB_CONV_MMA_SYNC) return GNB_EINVAL;
    int rc = unet_alloc_acts(u, 1);
    if (rc != GNB_OK) return rc;
    cudaMemsetAsync(u->xin, 0, (size_t)vox(u, 0, 1) * 16 * 2, u->s);
    u->tx_extra = 16;
    rc = unet_forward(u, 1);
    u->tx_extra = 0;
    return unet_check(u, rc);
}

int gnb_unet_test_set_plan(gnb_unet *u, int plan)
{
    if (!u || plan < -1) return GNB_EINVAL;
    int most = 0;
    for (auto &l : u->L) {
        if (l.kind != L_CONV3) continue;
        TcPlan plans[TC_MAX_PLANS];
        // (the coarsest grid's list is the shortest, the finest's the longest)
        most = std::max(most, conv3_tc_plans(l.Npad, l.Kpad, u->grid, plans, TC_MAX_PLANS));
        l.plan_f = plan;
    }
    new_generation(u);
    return most;
}

int gnb_unet_set_conv_impl(gnb_unet *u, int impl)
{
    if (!u || (impl != GNB_CONV_AUTO && impl != GNB_CONV_MMA_SYNC)) return GNB_EINVAL;
    u->conv_impl = impl;
    new_generation(u);
    return GNB_OK;
}

int gnb_unet_get_params(gnb_unet *u, float *dst, int on_device)
{
    if (!u || !dst) return GNB_EINVAL;
    cudaMemcpyAsync(dst, u->p, u->nparam * 4, on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost, u->s);
    return unet_check(u, GNB_OK);
}

int gnb_unet_get_grads(gnb_unet *u, float *dst, int on_device)
{
    if (!u || !dst) return GNB_EINVAL;
    cudaMemcpyAsync(dst, u->g, u->nparam * 4, on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost, u->s);
    return unet_check(u, GNB_OK);
}

int gnb_unet_get_activation(gnb_unet *u, int slot, int batch, float *dst, int on_device)
{
    if (!u || !dst || batch < 1 || batch > u->bcap || slot < 0) return GNB_EINVAL;
    // slot order: the input, then per level enc a, enc b (and the pooled
    // tensor below the coarsest level), then per decoder level (coarse to
    // fine) up, dec a, dec b
    const bf16 *src = nullptr;
    int C = 0, keep = 0, lev = 0;
    int k = slot;
    if (k == 0) {
        src = u->xin; C = 16; keep = u->cin; lev = 0;
    } else {
        k -= 1;
        for (int l = 0; l < u->levels && !src; l++) {
            const int w = width(u, l);
            const int nl = l + 1 < u->levels ? 3 : 2;
            if (k < nl) {
                src = u->act[k == 0 ? S_ENCA(l) : k == 1 ? S_ENCB(l) : S_POOL(l)];
                C = keep = w;
                lev = k == 2 ? l + 1 : l;
            }
            k -= nl;
        }
        for (int l = u->levels - 2; l >= 0 && !src; l--) {
            if (k < 3) {
                src = u->act[k == 0 ? S_UP(u, l) : k == 1 ? S_DECA(u, l) : S_DECB(u, l)];
                C = keep = width(u, l);
                lev = l;
            }
            k -= 3;
        }
    }
    if (!src) return GNB_EINVAL;
    const long long V = vox(u, lev, 1);
    const long long n = (long long)batch * V * keep;
    float *out = dst, *tmp = nullptr;
    if (!on_device) {
        if (cudaMalloc((void **)&tmp, n * 4) != cudaSuccess) {
            cudaGetLastError();
            return GNB_ENOMEM;
        }
        out = tmp;
    }
    counted(k_unblock)<<<(unsigned)((n + 255) / 256), 256, 0, u->s>>>(src, batch, C, V, keep, out);
    if (!on_device) cudaMemcpyAsync(dst, tmp, n * 4, cudaMemcpyDeviceToHost, u->s);
    int rc = unet_check(u, GNB_OK);
    if (tmp) cudaFree(tmp);
    return rc;
}

int gnb_unet_autotune(gnb_unet *u, int batch, double out_ms[2])
{
    if (!u || batch < 1) return GNB_EINVAL;
    int rc = unet_alloc_acts(u, batch);
    if (rc != GNB_OK) return rc;
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    if (cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess) {
        if (e0) cudaEventDestroy(e0);
        cudaGetLastError();
        return GNB_ECUDA;
    }
    auto timed = [&](double *ms) -> int {
        for (int w = 0; w < 2; w++) {
            int r = unet_forward(u, batch);
            if (r != GNB_OK) return r;
        }
        cudaEventRecord(e0, u->s);
        for (int w = 0; w < 3; w++) {
            int r = unet_forward(u, batch);
            if (r != GNB_OK) return r;
        }
        cudaEventRecord(e1, u->s);
        float f = 0.f;
        if (cudaEventSynchronize(e1) != cudaSuccess || cudaEventElapsedTime(&f, e0, e1) != cudaSuccess) return GNB_ECUDA;
        *ms = f / 3.0;
        return GNB_OK;
    };
    for (auto &ly : u->L) ly.plan_f = -1;
    double before = 0.0, after = 0.0;
    rc = timed(&before);
    if (rc == GNB_OK) {
        u->tuning = true;
        u->tuned_layers = 0;
        rc = unet_forward(u, batch);
        u->tuning = false;
    }
    if (rc == GNB_OK) rc = timed(&after);
    if (rc == GNB_OK && after > before)  // the timings of single layers did not add up: keep the rule
        for (auto &ly : u->L) ly.plan_f = -1;
    new_generation(u);
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    if (out_ms) {
        out_ms[0] = before;
        out_ms[1] = after;
    }
    return unet_check(u, rc);
}

int gnb_unet_get_output(gnb_unet *u, int batch, float *dst, int on_device)
{
    if (!u || !dst || batch < 1 || batch > u->bcap || !u->yout) return GNB_EINVAL;
    size_t bytes = (size_t)vox(u, 0, batch) * u->cout * 4;
    cudaMemcpyAsync(dst, u->yout, bytes, on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost, u->s);
    return unet_check(u, GNB_OK);
}

int gnb_unet_set_params(gnb_unet *u, const float *src, int on_device)
{
    if (!u || !src) return GNB_EINVAL;
    cudaMemcpyAsync(u->p, src, u->nparam * 4, on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice, u->s);
    cudaMemsetAsync(u->m, 0, u->nparam * 4, u->s);
    cudaMemsetAsync(u->v, 0, u->nparam * 4, u->s);
    u->adam_t = 0;
    return unet_check(u, unet_pack(u));
}

// Checkpoint of a network: a 64-byte header ("GNBUNET1", uint32 version 1,
// int32 cin, cout, base, levels, grid, int64 parameter count, int64 Adam
// steps taken, zero padding), then the FP32 master parameters and Adam's
// first and second moments, each [parameter count], in the order of
// gnb_unet_get_params.
namespace {
struct UnetCkHeader {
    char magic[8];
    uint32_t version;
    int32_t cin, cout, base, levels, grid;
    int64_t nparam, adam_t;
    unsigned char pad[64 - 8 - 4 - 20 - 16];
};
static_assert(sizeof(UnetCkHeader) == 64, "network checkpoint header is 64 bytes");
constexpr char UNET_MAGIC[8] = {'G', 'N', 'B', 'U', 'N', 'E', 'T', '1'};
}  // namespace

int gnb_unet_save(gnb_unet *u, const char *path)
{
    if (!u || !path) return GNB_EINVAL;
    std::vector<float> host((size_t)u->nparam * 3);
    for (int k = 0; k < 3; k++) {
        const float *src = k == 0 ? u->p : (k == 1 ? u->m : u->v);
        cudaMemcpyAsync(host.data() + (size_t)k * u->nparam, src, u->nparam * 4, cudaMemcpyDeviceToHost, u->s);
    }
    const int rc = unet_check(u, GNB_OK);
    if (rc != GNB_OK) return rc;
    UnetCkHeader h;
    memset(&h, 0, sizeof(h));
    memcpy(h.magic, UNET_MAGIC, 8);
    h.version = 1;
    h.cin = u->cin; h.cout = u->cout; h.base = u->base; h.levels = u->levels; h.grid = u->grid;
    h.nparam = u->nparam;
    h.adam_t = u->adam_t;
    FILE *f = fopen(path, "wb");
    if (!f) return GNB_EINVAL;
    const bool ok = fwrite(&h, sizeof(h), 1, f) == 1 && fwrite(host.data(), 4, host.size(), f) == host.size();
    const bool closed = fclose(f) == 0;
    return ok && closed ? GNB_OK : GNB_EINVAL;
}

int gnb_unet_load(gnb_unet *u, const char *path)
{
    if (!u || !path) return GNB_EINVAL;
    FILE *f = fopen(path, "rb");
    if (!f) return GNB_EINVAL;
    UnetCkHeader h;
    std::vector<float> host;
    int rc = GNB_OK;
    if (fread(&h, sizeof(h), 1, f) != 1 || memcmp(h.magic, UNET_MAGIC, 8) != 0 || h.version != 1) {
        rc = GNB_EINVAL;
    } else if (h.cin != u->cin || h.cout != u->cout || h.base != u->base || h.levels != u->levels ||
               h.grid != u->grid || h.nparam != u->nparam || h.adam_t < 0) {
        rc = GNB_EMISMATCH;
    } else {
        host.resize((size_t)u->nparam * 3);
        if (fread(host.data(), 4, host.size(), f) != host.size()) rc = GNB_EINVAL;
    }
    fclose(f);
    if (rc != GNB_OK) return rc;
    for (int k = 0; k < 3; k++) {
        float *dst = k == 0 ? u->p : (k == 1 ? u->m : u->v);
        cudaMemcpyAsync(dst, host.data() + (size_t)k * u->nparam, u->nparam * 4, cudaMemcpyHostToDevice, u->s);
    }
    u->adam_t = (int)h.adam_t;
    return unet_check(u, unet_pack(u));
}

int gnb_unet_forward(gnb_unet *u, int batch, const float *x, float *y, int on_device)
{
    if (!u || !x || !y || batch < 1) return GNB_EINVAL;
    int rc = unet_alloc_acts(u, batch);
    if (rc != GNB_OK) return rc;
    long long V = vox(u, 0, batch);
    const float *xd = x;
    float *tmpx = nullptr;
    if (!on_device) {
        if (cudaMalloc((void **)&tmpx, V * u->cin * 4) != cudaSuccess) return GNB_ENOMEM;
        cudaMemcpyAsync(tmpx, x, V * u->cin * 4, cudaMemcpyHostToDevice, u->s);
        xd = tmpx;
    }
    counted(k_pack_input)<<<batch_grid(vox(u, 0, 1), 256, batch), 256, 0, u->s>>>(xd, u->cin, batch, (int)vox(u, 0, 1),
                                                                                u->xin);
    rc = unet_forward(u, batch);
    if (rc == GNB_OK)
        cudaMemcpyAsync(y, u->yout, V * u->cout * 4, on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost,
                        u->s);
    rc = unet_check(u, rc);
    if (tmpx) cudaFree(tmpx);
    return rc;
}

int gnb_unet_train_step(gnb_unet *u, int batch, const float *x, const float *target, double lr, double *loss,
                        int on_device)
{
    if (!u || !x || !target || batch < 1 || !(lr >= 0.0)) return GNB_EINVAL;
    int rc = unet_alloc_acts(u, batch);
    if (rc != GNB_OK) return rc;
    long long V = vox(u, 0, batch);
    float *tmpx = nullptr;
    const float *xd = x;
    if (!on_device) {
        if (cudaMalloc((void **)&tmpx, V * u->cin * 4) != cudaSuccess) return GNB_ENOMEM;
        cudaMemcpyAsync(tmpx, x, V * u->cin * 4, cudaMemcpyHostToDevice, u->s);
        xd = tmpx;
    }
    cudaMemcpyAsync(u->tgt, target, V * u->cout * 4, on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice,
                    u->s);
    counted(k_pack_input)<<<batch_grid(vox(u, 0, 1), 256, batch), 256, 0, u->s>>>(xd, u->cin, batch, (int)vox(u, 0, 1),
                                                                                u->xin);
    rc = unet_forward(u, batch);
    cudaMemsetAsync(u->loss_d, 0, 8, u->s);
    counted(k_mse)<<<(unsigned)std::min((V + 255) / 256, 608LL), 256, 0, u->s>>>(u->yout, u->tgt, V, vox(u, 0, 1), u->cout,
                                                                     u->dyb, u->loss_d);
    cudaMemsetAsync(u->g, 0, u->nparam * 4, u->s);
    if (rc == GNB_OK) rc = unet_backward(u, batch);
    if (rc == GNB_OK && lr > 0.0) {
        u->adam_t++;
        const double b1 = 0.9, b2 = 0.999;
        const double ic1 = 1.0 / (1.0 - std::pow(b1, (double)u->adam_t));
        const double ic2 = 1.0 / (1.0 - std::pow(b2, (double)u->adam_t));
        counted(k_adam)<<<(unsigned)((u->nparam + 255) / 256), 256, 0, u->s>>>(
            u->p, u->g, u->m, u->v, u->nparam, (float)lr, (float)b1, (float)(1.0 - b1), (float)b2, (float)(1.0 - b2),
            1e-8f, (float)ic1, (float)ic2);
        rc = unet_pack(u);
    }
    double l = 0.0;
    if (rc == GNB_OK) cudaMemcpyAsync(&l, u->loss_d, 8, cudaMemcpyDeviceToHost, u->s);
    rc = unet_check(u, rc);
    if (loss) *loss = l / (double)(V * u->cout);
    if (tmpx) cudaFree(tmpx);
    return rc;
}

}  // extern "C"
