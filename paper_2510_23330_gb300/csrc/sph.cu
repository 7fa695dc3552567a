// sph.cu -- SPH kernel size, density/pressure and hydro force
// (Sec. 5.2.5, Table 3 "kernel size", "density and pressure", "hydro force"
// and Table 4 of Hirashima et al., SC'25).
//
// Kernel size: the support h_i of gas particle i is the distance to its
// n_ngb-th nearest gas neighbour (self included), neighbours ordered by
// (d^2, gas rank) with d^2 = (dx*dx + dy*dy) + dz*dz in FP64.  The paper
// iterates a search until it converges; here one warp takes a run of
// consecutive gas particles of one hydro-tree group and gathers every gas
// particle within a search radius R of the run into its shared memory, then
// selects the neighbours of one member after another:
//   1. FP32 distances d from FP32 offsets to the run's reference cell,
//      with |d - D| <= E(D) = 2^-23 (4 sqrt(3) A' sqrt(D) + 5 D), A' = the
//      largest offset in the run plus two grid units: each offset carries
//      one rounding (<= 2^-24 A') plus the residual's (<= 2^-24 unit), the
//      difference and the three fused multiply-adds one rounding each, and
//      the factor 2 over the first-order bound covers the second-order terms,
//   2. the candidates within the member's own radius (its previous support
//      times a margin: about 66 of them) are compacted into a list, and the
//      few largest removed one by one give the exact 64th smallest FP32
//      value t,
//   3. entries with d < t - 2E are certainly neighbours, entries with
//      d > t + 2E certainly not; only the few in between get the exact FP64
//      d^2 and are ranked by (d^2, gas rank).
// Members whose radius holds fewer than n_ngb particles are searched again
// with a larger one (from the count found, bisected once both bounds are
// known: the paper's "usually twice"); a run whose candidates do not fit is
// taken in smaller runs, and a single particle whose candidates do not fit is
// searched with a smaller radius, down to adjacent floats.  Density and the
// ideal-gas EOS are fused in.
//
// What bounds it: latency and instruction issue (50 % issue-active at 24 warps
// per SM, which the shared memory allows; HBM and L2 stay below 10 %).  A
// warp per run has no block barriers, and the compacted list replaces three
// passes over all candidates (histogram, bucket, classification) by one.
// Against one 128-thread CTA per group with those passes (phase time):
// 2^24 disk (1.68 M gas) 6.61 -> 3.07 ms, 2^20 disk (210 k) 1.03 -> 0.45 ms,
// 1e5-particle region 0.50 -> 0.27 ms, 4,096 gas 0.31 -> 0.05 ms.
//
// Force: symmetric SPH over S_i = N_i u {j : i in N_j}.  The reverse part is
// built from the non-mutual pairs only, so N_i and R_i are disjoint.
#include "common.cuh"

namespace gnb {

#define KN_THREADS 128
#define KN_WARPS (KN_THREADS / 32)
#define KN_CTAS 6     // CTAs per SM, as the shared memory of the warps allows
#define KN_CAP 448    // candidates of a warp's run
#define KN_STACK 384  // node stack entries of a warp
#define KN_LIST 128   // entries of one particle's list: 64 neighbours and at most 64 uncertain ones
#define KN_U 64
#define KN_GROUP 32   // gas particles of a hydro group
#define KN_GROW 1.03f // margin over the radius that the count within the last one asks for
#define KN_SUB 4      // particles per run when a run's candidates do not fit
#define NGB 64

__device__ __forceinline__ float kern_w(float r, float hinv)
{
    float q = r * hinv;
    float s = 2.546479089470325f * hinv * hinv * hinv;  // 8/pi h^-3
    if (q <= 0.5f) return s * (1.f - 6.f * q * q + 6.f * q * q * q);
    if (q <= 1.f) { float t = 1.f - q; return s * 2.f * t * t * t; }
    return 0.f;
}

__device__ __forceinline__ float kern_dw(float r, float hinv)
{
    float q = r * hinv;
    float s = 2.546479089470325f * hinv * hinv * hinv * hinv;
    if (q <= 0.5f) return s * (-12.f * q + 18.f * q * q);
    if (q <= 1.f) { float t = 1.f - q; return -6.f * s * t * t; }
    return 0.f;
}

// ---------------------------------------------------------------- gas extraction
struct GasGather {
    const uint64_t *skey;
    PArr p;
    int *gslot;
    int all;  // every particle is gas: slot k itself
    uint64_t *gkey;
    int *ggrank;
    int4 *C;
    float4 *R;
    float *gvx, *gvy, *gvz, *gu, *gRprev;
    double *gx, *gy, *gz;
    int ng;
    int pred;
    int have_h;
};

__global__ void k_gas_gather(GasGather g)
{
    int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= g.ng) return;
    int s = k;
    if (g.all) g.gslot[k] = k;
    else s = g.gslot[k];
    g.gkey[k] = g.skey[s];
    g.C[k] = make_int4(g.p.cx[s], g.p.cy[s], g.p.cz[s], __float_as_int(g.p.m[s]));
    g.R[k] = make_float4(g.p.rx[s], g.p.ry[s], g.p.rz[s], 0.f);
    g.gx[k] = g.p.x[s]; g.gy[k] = g.p.y[s]; g.gz[k] = g.p.z[s];
    g.ggrank[k] = g.p.grank[s];
    if (g.pred) {
        g.gvx[k] = g.p.vpx[s]; g.gvy[k] = g.p.vpy[s]; g.gvz[k] = g.p.vpz[s]; g.gu[k] = g.p.up[s];
    } else {
        g.gvx[k] = g.p.vx[s]; g.gvy[k] = g.p.vy[s]; g.gvz[k] = g.p.vz[s]; g.gu[k] = g.p.u[s];
    }
    g.gRprev[k] = g.have_h ? sqrtf((float)g.p.h2[s]) : 0.f;  // a starting radius only
}

// ---------------------------------------------------------------- work items
// A work item is a run of at most `sub` consecutive gas particles of one
// hydro group, with the starting search radius of the group where a particle
// has no previous support: from the density of the smallest ancestor cell
// holding at least n_ngb particles.
__global__ void k_knn_init(Tree t, int sub, const double *__restrict__ box, float *__restrict__ kR,
                           int2 *__restrict__ kitem, int *__restrict__ nitems)
{
    const int ng = *t.ngroups_d, lane = threadIdx.x & 31;
    const float unit = (float)box[4];
    for (int g0 = (blockIdx.x * blockDim.x + threadIdx.x) & ~31; g0 < ng; g0 += gridDim.x * blockDim.x) {
        const int g = g0 + lane;
        int4 a = make_int4(0, 0, 0, 0);
        float R = 0.f;
        if (g < ng) {
            int q = t.groups[g];
            a = t.na[q];
            int4 aq = a;
            while (aq.y < NGB && t.nb[q].w >= 0) {
                q = t.nb[q].w;
                aq = t.na[q];
            }
            R = 0.9f * (float)(1 << (GNB_MAXLEV - (aq.w & 255))) * unit * cbrtf((float)NGB / (float)max(aq.y, 1));
        }
        // items in group order within the warp, one atomic per warp; at most
        // one item per gas particle in all
        const int k = (a.y + sub - 1) / sub;
        int inc = k;
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += y;
        }
        int base = 0;
        if (lane == 31) base = atomicAdd(nitems, inc);
        base = __shfl_sync(0xffffffffu, base, 31) + inc - k;
        for (int e = 0; e < k; e++) {
            kitem[base + e] = make_int2(a.x + e * sub, min(sub, a.y - e * sub));
            kR[base + e] = R;
        }
    }
}

struct KnnParams {
    const int4 *na, *nb;  // hydro tree
    const int2 *item;
    const float *kR;
    const int *nitems;
    int *next;           // next item to take
    int *nunder;         // items whose radius held too few candidates for some member
    const int4 *C;       // cell x, y, z and mass bits per gas particle
    const float4 *R;     // residual x, y, z
    const int *ggrank;
    const float *gu;
    const double *gx, *gy, *gz;
    const double *box;
    const float *rprev;  // previous support per gas particle (0: none)
    float margin;        // search radius over the previous support
    int *failed;         // set when a particle could not be ranked
    int *nbr;
    float *nd2;
    double *h2;
    float2 *h2b;         // h^2 rounded down and up to FP32
    float *h, *E;
    int *g64;
    const float *gvx, *gvy, *gvz;
    float4 *V, *Q;       // records of the force pass (see pair_force)
    const int *gslot;    // particle slot of each gas particle, and the fields per slot
    float *s_rho, *s_pres, *s_cs;
    float gamma;
    int pressure;  // 1: also smooth P = (gamma - 1) sum_j m_j u_j W_ij (pressure-energy SPH)
};

// Per-warp buffers: the candidates, and a scratch area that holds the node
// stack and the pending leaves during the walk, then the particle's list and
// its uncertain entries.
struct KnnWarp {
    float4 cand[KN_CAP];
    union {
        struct {
            unsigned stack[KN_STACK];
            int2 leaf[64];
        } walk;
        struct {
            float d[KN_LIST];
            int j[KN_LIST];
            long long uD[KN_U];  // exact FP64 d^2 as bit patterns (non-negative: they order like the values)
            int uj[KN_U];
            int ug[KN_U];        // gas ranks of the uncertain entries
        } sel;
    };
};

__device__ __forceinline__ float d2f(float4 c, float xi, float yi, float zi)
{
    float dx = c.x - xi, dy = c.y - yi, dz = c.z - zi;
    return __fmaf_rn(dx, dx, __fmaf_rn(dy, dy, dz * dz));
}

__device__ __forceinline__ double exact_d2(const double *x, const double *y, const double *z, int i, int j)
{
    double dx = __dsub_rn(x[i], x[j]), dy = __dsub_rn(y[i], y[j]), dz = __dsub_rn(z[i], z[j]);
    double a = __dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy));
    return __dadd_rn(a, __dmul_rn(dz, dz));
}

// Box of a run of particles (cells [b0, b1]), its reference cell, and the box
// in offset coordinates [lo, hi).
struct KnnBox {
    int b0[3], b1[3], gref[3];
    float lo[3], hi[3];
};

// Candidates of a warp's batch of m <= 32 leaves (lane q holds leaf q: first
// and count): the particles of the leaves side by side, 32 at a time.  Lane f
// of a chunk finds its leaf from the leaf starts in the chunk (one bit each)
// and the number of leaves that start before it.  Returns false when the
// buffer is full.  one (the run is a single particle at xs): the distance to
// it decides rather than the box.
__device__ __forceinline__ bool knn_gather(KnnWarp &S, const KnnParams &p, const KnnBox &B, int m, int2 leaf, float unit,
                                           float R2stage, bool one, float xs, float ys, float zs, int &nc,
                                           float &amax, int lane)
{
    const unsigned ltmask = (1u << lane) - 1u, lemask = ltmask | (1u << lane);
    const int cnt = lane < m ? leaf.y : 0;
    int inc = cnt;
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += y;
    }
    const int total = __shfl_sync(0xffffffffu, inc, 31);
    const int start = lane < m ? inc - cnt : 0x3fffffff;
    const int rel = leaf.x - start;
    for (int c = 0; c < total; c += 32) {
        const unsigned st = (unsigned)(start - c);
        const unsigned mask = __reduce_or_sync(0xffffffffu, st < 32u ? 1u << st : 0u);
        const int before = __popc(__ballot_sync(0xffffffffu, start < c));
        const int ord = before + __popc(mask & lemask) - 1;
        const int j = __shfl_sync(0xffffffffu, rel, ord) + c + lane;
        bool in = false;
        float ox = 0.f, oy = 0.f, oz = 0.f;
        if (c + lane < total) {
            const int4 C = __ldg(&p.C[j]);
            const float4 r = __ldg(&p.R[j]);
            ox = grid_off(C.x, B.gref[0], r.x, unit);
            oy = grid_off(C.y, B.gref[1], r.y, unit);
            oz = grid_off(C.z, B.gref[2], r.z, unit);
            if (one) {
                in = d2f(make_float4(ox, oy, oz, 0.f), xs, ys, zs) <= R2stage;
            } else {
                const float gx = fmaxf(0.f, fmaxf(B.lo[0] - ox, ox - B.hi[0]));
                const float gy = fmaxf(0.f, fmaxf(B.lo[1] - oy, oy - B.hi[1]));
                const float gz = fmaxf(0.f, fmaxf(B.lo[2] - oz, oz - B.hi[2]));
                in = gx * gx + gy * gy + gz * gz <= R2stage;
            }
        }
        const unsigned bal = __ballot_sync(0xffffffffu, in);
        const int add = __popc(bal);
        if (nc + add > KN_CAP) return false;
        if (in) {
            S.cand[nc + __popc(bal & ltmask)] = make_float4(ox, oy, oz, __int_as_float(j));
            amax = fmaxf(amax, ox * ox + oy * oy + oz * oz);
        }
        nc += add;
    }
    return true;
}

// Walk of the hydro tree: every particle within R of the run's box (of the
// particle, for a run of one) becomes a candidate.  The stack holds nodes
// whose children are to be tested, as (first child << 3) | (children - 1)
// (node indices below 2^29, checked by the host); a round tests the children
// of up to four of them, eight lanes each, so a push is one ballot and one
// store.  False when the candidate buffer is full.
__device__ __forceinline__ bool knn_walk(KnnWarp &S, const KnnParams &p, const KnnBox &B, float R, float unit, bool one,
                                         float xs, float ys, float zs, int &nc, float &amax, int lane)
{
    const unsigned ltmask = (1u << lane) - 1u;
    // node test in grid units, only a bound for the particle tests below:
    // gaps are integers below 2^22, exact in FP32, and the margin covers the
    // roundings of the sums
    const float Rg = R / unit;  // unit is a power of two
    const float Rg2 = Rg * Rg * (1.f + 1e-5f) + 4.f;
    // a single particle keeps what can lie in its list: d^2 <= R^2 + 2 E, with a
    // margin (E < 2^-23 (12 R^2 + 26 unit R) there: A' is at most R, sqrt(3)
    // units to the particle and two more; 2 E < 2.9e-6 R^2 + 6.2e-6 unit R,
    // below the margin by (1.1 R^2 - 0.2 unit R + 6 unit^2) 1e-6 > 0)
    const float R2stage = one ? R * R * (1.f + 4e-6f) + 6e-6f * unit * (R + unit)
                              : R * R * (1.f + 1e-4f) + 4.f * unit * unit;
    nc = 0;
    amax = 0.f;
    int sp = 0, nl = 0;
    // the first round tests the root alone
    int node = lane == 0 ? 0 : -1;
    for (;;) {
        int nch = 0, child = 0, first = 0, count = 0;
        if (node >= 0) {
            const int4 a = __ldg(&p.na[node]);
            const int4 C = __ldg(&p.nb[node]);
            const int s = 1 << (GNB_MAXLEV - (a.w & 255));
            const float gx = (float)max(0, max(C.x - (B.b1[0] + 1), B.b0[0] - (C.x + s)));
            const float gy = (float)max(0, max(C.y - (B.b1[1] + 1), B.b0[1] - (C.y + s)));
            const float gz = (float)max(0, max(C.z - (B.b1[2] + 1), B.b0[2] - (C.z + s)));
            if (gx * gx + gy * gy + gz * gz <= Rg2) {
                nch = a.w >> 8;
                child = a.z;
                first = a.x;
                if (nch == 0) count = a.y;
            }
        }
        __syncwarp();
        const unsigned pb = __ballot_sync(0xffffffffu, nch > 0), lb = __ballot_sync(0xffffffffu, count > 0);
        if (nch > 0) S.walk.stack[sp + __popc(pb & ltmask)] = (unsigned)child << 3 | (unsigned)(nch - 1);
        if (count > 0) S.walk.leaf[nl + __popc(lb & ltmask)] = make_int2(first, count);
        sp += __popc(pb);
        nl += __popc(lb);
        __syncwarp();
        if (nl >= 32 || (sp == 0 && nl > 0)) {
            const int m = min(nl, 32);
            nl -= m;
            const int2 lf = lane < m ? S.walk.leaf[nl + lane] : make_int2(0, 0);
            if (!knn_gather(S, p, B, m, lf, unit, R2stage, one, xs, ys, zs, nc, amax, lane)) return false;
        }
        if (sp == 0) {
            if (nl == 0) return true;
            node = -1;
            continue;
        }
        // up to four nodes while the stack is at most half full (a round then
        // leaves at most 28 more entries), else one (seven more per level below
        // it, at most GNB_MAXLEV levels): it cannot overflow
        static_assert(KN_STACK / 2 + 28 + 7 * GNB_MAXLEV <= KN_STACK, "walk stack");
        const int k = sp <= KN_STACK / 2 ? min(4, sp) : 1;
        const int q = lane >> 3;
        const unsigned e = q < k ? S.walk.stack[sp - k + q] : 0u;
        node = q < k && (lane & 7) <= (int)(e & 7u) ? (int)(e >> 3) + (lane & 7) : -1;
        sp -= k;
    }
}

enum { KN_DONE = 0, KN_UNDER = 1, KN_FAIL = 2 };

// Candidates of particle (xi, yi, zi) with d^2 <= T, compacted into the list
// (the first KN_LIST of them); returns their number.
__device__ __forceinline__ int knn_list(KnnWarp &S, int nc, float xi, float yi, float zi, float T, int lane)
{
    const unsigned ltmask = (1u << lane) - 1u;
    int n = 0;
    __syncwarp();
    for (int c0 = 0; c0 < nc; c0 += 32) {
        const int c = c0 + lane;
        float d = 3.0e38f;
        int j = 0;
        if (c < nc) {
            const float4 v = S.cand[c];
            d = d2f(v, xi, yi, zi);
            j = __float_as_int(v.w);
        }
        const bool in = d <= T;
        const unsigned bal = __ballot_sync(0xffffffffu, in);
        const int pos = n + __popc(bal & ltmask);
        if (in && pos < KN_LIST) {
            S.sel.d[pos] = d;
            S.sel.j[pos] = j;
        }
        n += __popc(bal);
    }
    __syncwarp();
    return n;
}

__device__ __forceinline__ float sqrt_fast(float x)
{
    float r;
    asm("sqrt.approx.f32 %0, %1;" : "=f"(r) : "f"(x));  // relative error below 2^-22
    return r;
}

// What the selection of one particle leaves to its lane: its 64th neighbour
// (-1: ranked already, hsq holds its exact d^2) and the FP32 error bound.
struct KnnSel {
    int j64, g64;
    float E;
    double hsq;
};

// The 64 nearest of particle i among the candidates, exactly (see the file
// comment): fewer than 64 with d^2 <= thr is KN_UNDER, T0 is the largest d^2
// that can matter.  The list goes to nbr / nd2 except, in the usual case of
// one uncertain entry, its last place (r.j64).  n: entries of the last list
// (KN_UNDER: about how many lie within the radius).
__device__ __forceinline__ int knn_select(KnnWarp &S, const KnnParams &p, int i, int nc, float xi, float yi, float zi,
                                          float thr, float T0, float EA, int &n, KnnSel &r, int lane)
{
    constexpr float U = 1.1920929e-07f;  // 2^-23
    constexpr int KPL = KN_LIST / 32;
    const unsigned ltmask = (1u << lane) - 1u;
    float T = T0, Tlo = 0.f, Thi = T0;  // Tlo: too few entries, Thi: too many
    float t = 0.f, E = 0.f;
    bool band = false;  // T is the upper end of the uncertain band
    unsigned du[KPL];
    for (int it = 0;; it++) {
        n = knn_list(S, nc, xi, yi, zi, T, lane);
        if (n < NGB && it == 0) return KN_UNDER;
        // fewer than 64 lie below the band, so more than KN_U of the list's
        // entries are in it: narrowing would find the same t and band again
        if (n > KN_LIST && band) return KN_FAIL;
        if (n < NGB || n > KN_LIST) {
            // more than the list holds within the radius: narrow it to 64 ..
            // KN_LIST entries, by the number density, then by bisection down
            // to adjacent floats
            if (n > KN_LIST) Thi = T;
            else Tlo = T;
            float q = T * __powf(88.f / (float)max(n, 1), 0.6666667f);
            if (it >= 6 || !(q > Tlo && q < Thi)) q = 0.5f * (Tlo + Thi);
            if (!(q > Tlo && q < Thi) || it >= 64) return KN_FAIL;
            T = q;
            continue;
        }
        // t = the 64th smallest: the largest after n - 64 removals, or, when
        // the list holds many more, bit by bit (float bits order like values)
#pragma unroll
        for (int k = 0; k < KPL; k++) {
            const int e = lane + 32 * k;
            du[k] = e < n ? __float_as_uint(S.sel.d[e]) : 0u;
        }
        unsigned tb = 0u;
        if (n - NGB <= 20) {
            unsigned w[KPL];
#pragma unroll
            for (int k = 0; k < KPL; k++) w[k] = du[k];
            for (int r = n - NGB;; r--) {
                unsigned m = w[0];
#pragma unroll
                for (int k = 1; k < KPL; k++) m = max(m, w[k]);
                tb = __reduce_max_sync(0xffffffffu, m);
                if (r == 0) break;
                const unsigned who = __ballot_sync(0xffffffffu, m == tb);
                if (lane == __ffs(who) - 1) {
                    bool gone = false;
#pragma unroll
                    for (int k = 0; k < KPL; k++)
                        if (!gone && w[k] == tb) { w[k] = 0u; gone = true; }
                }
            }
        } else {
            // the largest v with fewer than 64 entries below it
#pragma unroll 1
            for (int b = 30; b >= 0; b--) {
                const unsigned v = tb | (1u << b);
                int c = 0;
#pragma unroll
                for (int k = 0; k < KPL; k++) c += (lane + 32 * k < n && du[k] < v) ? 1 : 0;
                if (__reduce_add_sync(0xffffffffu, c) < NGB) tb = v;
            }
        }
        t = __uint_as_float(tb);
        if (t > thr) return KN_UNDER;  // fewer than 64 certainly within R
        // the bound at a point just above the band's upper end (E << t)
        const float te = t * 1.0009765625f;
        E = U * (EA * sqrt_fast(te) + 5.f * te);
        if (t + 2.f * E <= T) break;
        T = t + 2.f * E;  // the band reaches past a narrowed radius
        band = true;
    }
    const float lo = t - 2.f * E, hi = t + 2.f * E;
    // sure members (fewer than 64 lie below t) to the list, uncertain ones
    // collected
    int *outn = p.nbr + (size_t)i * NGB;
    float *outd = p.nd2 + (size_t)i * NGB;
    int nS = 0, nu = 0, ju = 0;
#pragma unroll
    for (int k = 0; k < KPL; k++) {
        if (32 * k < n) {  // (uniform)
            const bool have = lane + 32 * k < n;
            const float d = __uint_as_float(du[k]);
            const int j = have ? S.sel.j[lane + 32 * k] : 0;
            const bool sure = have && d < lo, unc = have && !sure && d <= hi;
            const unsigned sb = __ballot_sync(0xffffffffu, sure), ub = __ballot_sync(0xffffffffu, unc);
            if (sure) {
                const int pos = nS + __popc(sb & ltmask);
                outn[pos] = j;
                outd[pos] = d;
            }
            if (unc) {
                const int pos = nu + __popc(ub & ltmask);
                if (pos < KN_U) S.sel.uj[pos] = j;
            }
            nS += __popc(sb);
            nu += __popc(ub);
        }
    }
    r.E = E;
    if (nu > KN_U) return KN_FAIL;
    __syncwarp();
    if (nu == 1) {  // t itself: nS is 63
        r.j64 = S.sel.uj[0];
        return KN_DONE;
    }
    const int need = NGB - nS;
    double hsq = 0.0;
    int h64 = -1;
    bool have = false;
#pragma unroll 1
    for (int e = lane; e < nu; e += 32) {
        const int je = S.sel.uj[e];
        S.sel.uD[e] = __double_as_longlong(exact_d2(p.gx, p.gy, p.gz, i, je));
        S.sel.ug[e] = p.ggrank[je];
    }
    __syncwarp();
#pragma unroll 1
    for (int e = lane; e < nu; e += 32) {
        const long long De = S.sel.uD[e];
        const int ge = S.sel.ug[e];
        int rk = 0;
#pragma unroll 1
        for (int f = 0; f < nu; f++) {  // integer compares: no FP64 work
            const long long Df = S.sel.uD[f];
            rk += (Df < De) || (Df == De && S.sel.ug[f] < ge);
        }
        if (rk < need) {
            outn[nS + rk] = S.sel.uj[e];
            outd[nS + rk] = (float)__longlong_as_double(De);
        }
        if (rk == need - 1) { hsq = __longlong_as_double(De); h64 = ge; have = true; }
    }
    const unsigned hb = __ballot_sync(0xffffffffu, have);
    if (hb == 0u) return KN_FAIL;  // error bound violated: fewer uncertain entries than needed
    const int hs = __ffs(hb) - 1;
    r.hsq = __shfl_sync(0xffffffffu, hsq, hs);
    r.g64 = __shfl_sync(0xffffffffu, h64, hs);
    r.j64 = -1;
    return KN_DONE;
}

// The results of the members `done` of a run whose neighbours are selected
// (lane k: member k, particle first + k, its selection in r): the exact
// support, lane by lane, then each member's density and pressure sums over
// the warp, then the equation of state, again lane by lane.
__device__ __forceinline__ void knn_finish(const KnnParams &p, int first, unsigned done, const KnnSel &r, int lane)
{
    const bool mine = (done >> lane) & 1u;
    const int i = first + lane;
    float hinv = 0.f;
    if (mine) {
        double hsq = r.hsq;
        int g64 = r.g64;
        if (r.j64 >= 0) {
            hsq = exact_d2(p.gx, p.gy, p.gz, i, r.j64);
            g64 = p.ggrank[r.j64];
            p.nbr[(size_t)i * NGB + NGB - 1] = r.j64;
            p.nd2[(size_t)i * NGB + NGB - 1] = (float)hsq;
        }
        const float hh = sqrtf((float)hsq);  // within one FP32 rounding of sqrt(h^2)
        hinv = 1.f / hh;
        p.h2[i] = hsq;
        p.h2b[i] = make_float2(__double2float_rd(hsq), __double2float_ru(hsq));
        p.h[i] = hh;
        p.g64[i] = g64;
        p.E[i] = r.E;
    }
    __syncwarp();
    float rho = 0.f, qsum = 0.f;
#pragma unroll 1
    for (unsigned m = done; m; m &= m - 1u) {
        const int k = __ffs(m) - 1;
        const float hk = __shfl_sync(0xffffffffu, hinv, k);
        const int *nb = p.nbr + (size_t)(first + k) * NGB;
        const float *nd = p.nd2 + (size_t)(first + k) * NGB;
        float rs = 0.f, qs = 0.f;
#pragma unroll
        for (int q = 0; q < NGB / 32; q++) {
            const int j = nb[lane + 32 * q];
            const float mw = __int_as_float(p.C[j].w) * kern_w(sqrtf(nd[lane + 32 * q]), hk);
            rs += mw;
            if (p.pressure) qs = __fmaf_rn(mw, p.gu[j], qs);
        }
        rs = warp_sum(rs);
        if (p.pressure) qs = warp_sum(qs);
        if (lane == k) { rho = rs; qsum = qs; }
    }
    if (mine) {
        const float u = p.gu[i];
        const float P = p.pressure ? (p.gamma - 1.f) * qsum : (p.gamma - 1.f) * rho * u;
        const float cs = sqrtf(p.gamma * P / rho);
        const int s = p.gslot[i];
        p.s_rho[s] = rho;
        p.s_pres[s] = P;
        p.s_cs[s] = cs;
        p.V[i] = make_float4(p.gvx[i], p.gvy[i], p.gvz[i], cs);
        if (p.pressure) {
            const float U = (p.gamma - 1.f) * u;
            p.Q[i] = make_float4(rho, U / P, U, hinv);
        } else {
            p.Q[i] = make_float4(rho, P / (rho * rho), 1.f, hinv);
        }
    }
}

// Kernel-size search of the run [first, first + len), len <= 32, from radius
// R0 (see the file comment).  KN_FAIL: some member could not be ranked within
// the buffers.
__device__ __forceinline__ int knn_run(KnnWarp &S, const KnnParams &p, int first, int len, float R0, float unit,
                                       bool &widened, int lane)
{
    KnnBox B;
    const bool mine = lane < len;
    int4 C = make_int4(0, 0, 0, 0);
    float4 r = make_float4(0.f, 0.f, 0.f, 0.f);
    float hp = 0.f;
    if (mine) {
        C = p.C[first + lane];
        r = p.R[first + lane];
        hp = p.rprev[first + lane];
    }
    const int cc[3] = {C.x, C.y, C.z};
#pragma unroll
    for (int a = 0; a < 3; a++) {
        B.b0[a] = __reduce_min_sync(0xffffffffu, mine ? cc[a] : 0x7fffffff);
        B.b1[a] = __reduce_max_sync(0xffffffffu, mine ? cc[a] : -1);
        B.gref[a] = (B.b0[a] + B.b1[a]) >> 1;
        B.lo[a] = (float)(B.b0[a] - B.gref[a]) * unit;
        B.hi[a] = (float)(B.b1[a] + 1 - B.gref[a]) * unit;
    }
    const float xo = grid_off(C.x, B.gref[0], r.x, unit);
    const float yo = grid_off(C.y, B.gref[1], r.y, unit);
    const float zo = grid_off(C.z, B.gref[2], r.z, unit);
    const bool known = __all_sync(0xffffffffu, !mine || hp > 0.f);
    const unsigned hmax = __reduce_max_sync(0xffffffffu, __float_as_uint(hp));
    float R = known ? p.margin * __uint_as_float(hmax) : R0;
    const float xs = __shfl_sync(0xffffffffu, xo, 0), ys = __shfl_sync(0xffffffffu, yo, 0),
                zs = __shfl_sync(0xffffffffu, zo, 0);
    unsigned todo = len == 32 ? 0xffffffffu : (1u << len) - 1u;
    float Rlo = 0.f, Rhi = 0.f;  // radii known to be too small and too large
    for (int it = 0; it < 96; it++) {
        int nc;
        float amax;
        if (!knn_walk(S, p, B, R, unit, len == 1, xs, ys, zs, nc, amax, lane)) {
            if (len > 1) return KN_FAIL;
            Rhi = R;
            R = Rlo > 0.f ? 0.5f * (R + Rlo) : 0.6f * R;
            if (!(R > Rlo && R < Rhi)) return KN_FAIL;
            continue;
        }
        // the run's own particles also bound the offsets
        if (mine) amax = fmaxf(amax, xo * xo + yo * yo + zo * zo);
        amax = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(amax)));
        // error bound of an FP32 d^2 near D (see the file comment)
        const float EA = 6.92820323f * (sqrtf(amax) + 2.f * unit);  // 4 sqrt(3) A'
        // lane k: member k's radius (its own previous support's, or R), thr
        // and T0: fewer than 64 with d^2 <= thr lie certainly within it, and
        // t + 2 E(t) <= T0 for every t <= thr
        unsigned left = 0u, done = 0u;
        float grow = 1.f;  // the factor by which R falls short, from the counts within it
        KnnSel sel;
        sel.j64 = -1; sel.g64 = 0; sel.E = 0.f; sel.hsq = 0.0;
        const float Rk = hp > 0.f ? fminf(R, p.margin * hp) : R;
        unsigned m = todo;
        bool wide = false;  // the member found too few within its own radius: now within R
#pragma unroll 1
        while (m) {
            const int k = __ffs(m) - 1;
            const float rk = __shfl_sync(0xffffffffu, Rk, k), Ri = wide ? R : rk;
            const float xi = __shfl_sync(0xffffffffu, xo, k), yi = __shfl_sync(0xffffffffu, yo, k),
                        zi = __shfl_sync(0xffffffffu, zo, k);
            constexpr float U = 1.1920929e-07f;  // 2^-23
            const float R2 = Ri * Ri;
            const float thr = R2 - U * (EA * Ri + 5.f * R2);
            const float T0 = R2 + 2.f * U * (EA * (Ri * 1.0005f) + 5.01f * R2);
            KnnSel one;
            int n = 0;
            const int rc = knn_select(S, p, first + k, nc, xi, yi, zi, thr, T0, EA, n, one, lane);
            if (rc == KN_FAIL) return KN_FAIL;
            if (rc == KN_UNDER && Ri < R) {
                wide = true;
                continue;
            }
            if (rc == KN_UNDER) {
                left |= 1u << k;
                grow = fmaxf(grow, KN_GROW * cbrtf((float)NGB / (float)max(min(n, NGB), 1)));
            } else {
                done |= 1u << k;
                if (lane == k) sel = one;
            }
            wide = false;
            m &= m - 1u;
        }
        knn_finish(p, first, done, sel, lane);
        if (left == 0u) return KN_DONE;
        widened = true;
        todo = left;
        Rlo = R;
        R = Rhi > 0.f ? 0.5f * (R + Rhi) : fminf(grow, 1.6f) * R;
        if (Rhi > 0.f && !(R > Rlo && R < Rhi)) return KN_FAIL;
    }
    return KN_FAIL;
}

__global__ void __launch_bounds__(KN_THREADS, KN_CTAS) k_knn(KnnParams p)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    KnnWarp &S = reinterpret_cast<KnnWarp *>(smem_raw)[threadIdx.x >> 5];
    const int lane = threadIdx.x & 31;
    const float unit = (float)p.box[4];
    const int nitems = *p.nitems;
    for (;;) {
        int it = 0;
        if (lane == 0) it = atomicAdd(p.next, 1);
        it = __shfl_sync(0xffffffffu, it, 0);
        if (it >= nitems) break;
        const int2 item = p.item[it];
        const float R0 = p.kR[it];
        bool widened = false;
        const int end = item.x + item.y;
        int step = item.y;
        for (int pos = item.x; pos < end;) {
            const int len = min(step, end - pos);
            if (knn_run(S, p, pos, len, R0, unit, widened, lane) == KN_DONE) {
                pos += len;
            } else if (len > 1) {
                // the members do not fit the buffers together: smaller runs
                // (each with the radius of its own members), then singles
                step = len > KN_SUB ? KN_SUB : 1;
            } else {
                if (lane == 0) atomicOr(p.failed, 1);
                pos++;
            }
        }
        if (widened && lane == 0) atomicAdd(p.nunder, 1);
    }
}

// ---------------------------------------------------------------- symmetric lists
// Bit k of mut[i] is set when entry k of N_i is mutual (i in N_j too), using
// (d^2, gas rank) <= (h_j^2, rank of j's n_ngb-th neighbour).  The FP32 d^2
// lies within 2 E_i of the FP64 one; the interval [d - 2E, d + 2E], widened
// by directed rounding, is first compared with h_j^2 rounded down and up to
// FP32 (no FP64 work: GB300 issues FP64 at a small fraction of the FP32
// rate).  Only a pair that test leaves open takes the FP64 test and, within
// its band, the exact FP64 d^2.  Every decision the FP32 test takes is the
// one the FP64 test would take.
//
// The particles' supports are stored here too.
//
// SL lanes share a particle here and in the list fill: a lane takes every
// SL-th entry, so a row of the list is read in whole sectors and the gathers
// of a particle overlap (one thread per particle: a chain of 64 reads).
template <int SL>
__global__ void __launch_bounds__(256) k_mutual(int ng, const int *__restrict__ nbr, const float *__restrict__ nd2,
                                                const float *__restrict__ E, const double *__restrict__ h2,
                                                const float2 *__restrict__ h2b, const int *__restrict__ g64,
                                                const int *__restrict__ grank, const double *__restrict__ x,
                                                const double *__restrict__ y, const double *__restrict__ z,
                                                unsigned long long *__restrict__ mut, int *__restrict__ rcnt,
                                                int *__restrict__ rtot, const int *__restrict__ gslot,
                                                double *__restrict__ s_h2)
{
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t == 0) *rtot = 0;  // summed by k_rev_off
    const int i = t / SL, l = threadIdx.x & (SL - 1), half = (threadIdx.x & 31) / SL;
    const bool valid = i < ng;
    unsigned long long mask = 0ull;
    const float Ei = valid ? E[i] : 0.f;
    const float e2 = 2.f * Ei;  // exact
    int jk[NGB / SL];
    float dk[NGB / SL];
#pragma unroll
    for (int q = 0; q < NGB / SL; q++) {
        jk[q] = valid ? nbr[(size_t)i * NGB + q * SL + l] : 0;
        dk[q] = valid ? nd2[(size_t)i * NGB + q * SL + l] : 0.f;
    }
#pragma unroll
    for (int q = 0; q < NGB / SL; q++) {
        const int j = jk[q];
        const float df = dk[q];
        bool m = true;
        if (valid && j != i) {
            const float2 hb = h2b[j];
            if (__fadd_ru(df, e2) < hb.x) m = true;
            else if (__fsub_rd(df, e2) > hb.y) m = false;
            else {
                double d = (double)df;
                double hj = h2[j];
                double e = 2.0 * (double)Ei;
                if (d + e < hj) m = true;
                else if (d - e > hj) m = false;
                else {
                    double D = exact_d2(x, y, z, i, j);
                    m = (D < hj) || (D == hj && grank[i] <= g64[j]);
                }
            }
            if (!m) atomicAdd(&rcnt[j], 1);
        }
        const unsigned bal = __ballot_sync(0xffffffffu, m);
        mask |= (unsigned long long)((bal >> (SL * half)) & ((1u << SL) - 1u)) << (q * SL);
    }
    if (valid && l == 0) {
        mut[i] = mask;
        s_h2[gslot[i]] = h2[i];  // see sph_keep_support
    }
}

// Storage of the reverse lists: each particle's segment of rlist, taken in
// blocks of a warp's particles from a running total (their order does not
// matter, so no scan over all particles is needed).
__global__ void __launch_bounds__(256) k_rev_off(int ng, const int *__restrict__ rcnt, int *__restrict__ roff,
                                                 int *__restrict__ rcur, int *__restrict__ rtot)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x, lane = threadIdx.x & 31;
    const int v = i < ng ? rcnt[i] : 0;
    int inc = v;
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += y;
    }
    int base = 0;
    if (lane == 31 && inc > 0) base = atomicAdd(rtot, inc);
    base = __shfl_sync(0xffffffffu, base, 31) + inc - v;
    if (i < ng) {
        roff[i] = base;
        rcur[i] = base;
    }
}

template <int SL>
__global__ void __launch_bounds__(256) k_rev_fill(int ng, const int *__restrict__ nbr,
                                                  const unsigned long long *__restrict__ mut, int *__restrict__ rcur,
                                                  int *__restrict__ rlist)
{
    const int i = (blockIdx.x * blockDim.x + threadIdx.x) / SL, l = threadIdx.x & (SL - 1);
    if (i >= ng) return;
    const unsigned long long mask = mut[i];
#pragma unroll
    for (int q = 0; q < NGB / SL; q++) {
        if (mask & (1ull << (q * SL + l))) continue;
        const int j = nbr[(size_t)i * NGB + q * SL + l];
        rlist[atomicAdd(&rcur[j], 1)] = i;
    }
}

// ---------------------------------------------------------------- force
struct ForceParams {
    int ng;
    const int *nbr, *roff, *rcnt, *rlist;
    const int4 *C;    // neighbour records (gas gather and kernel-size search)
    const float4 *R, *V, *Q;
    const double *box;
    float alpha;
    const int *gslot;
    float *ax, *ay, *az, *dudt;  // per particle slot: the hydro part is added to the acceleration
    float *vsig;  // largest signal velocity c_i + c_j - 3 min(w_ij, 0) over the pairs of i
};

// One record set per gas particle so a pair gathers four records instead of
// fourteen fields: {cell, mass}, {residual}, {v, c}, {rho, Y, U, 1/h}.  The
// pressure terms of a pair are U_j Y_i gW(h_i) + U_i Y_j gW(h_j): Y = P/rho^2,
// U = 1 for density-energy SPH; Y = (gamma-1) u / P, U = (gamma-1) u for
// pressure-energy SPH with the smoothed P, whose pair coefficients are
// (gamma-1)^2 u_i u_j / P_i and / P_j.
__device__ __forceinline__ void pair_force(const ForceParams &p, int j, float unit, int ci0, int ci1, int ci2,
                                           float ri0, float ri1, float ri2, float vi0, float vi1, float vi2,
                                           float hinv_i, float pi_, float ui_, float rhoi, float csi, float &a0,
                                           float &a1, float &a2, float &du, float &vs)
{
    const int4 Cj = p.C[j];
    const float4 Rj = p.R[j];
    const float4 Vj = p.V[j];
    const float4 Qj = p.Q[j];
    float dx = __fmaf_rn((float)(ci0 - Cj.x), unit, ri0 - Rj.x);
    float dy = __fmaf_rn((float)(ci1 - Cj.y), unit, ri1 - Rj.y);
    float dz = __fmaf_rn((float)(ci2 - Cj.z), unit, ri2 - Rj.z);
    float r2 = __fmaf_rn(dx, dx, __fmaf_rn(dy, dy, dz * dz));
    float r = sqrtf(r2);
    float rinv = r > 0.f ? 1.f / r : 0.f;
    float dwi = kern_dw(r, hinv_i), dwj = kern_dw(r, Qj.w);
    float rhoj = Qj.x;
    float pj_ = Qj.y;
    float vx = vi0 - Vj.x, vy = vi1 - Vj.y, vz = vi2 - Vj.z;
    float w = (vx * dx + vy * dy + vz * dz) * rinv;
    float visc = 0.f;
    float vsig = csi + Vj.w - 3.f * fminf(w, 0.f);
    vs = fmaxf(vs, vsig);
    if (w < 0.f) visc = -0.5f * p.alpha * vsig * w / (0.5f * (rhoi + rhoj));
    float dwbar = 0.5f * (dwi + dwj);
    float mj = __int_as_float(Cj.w);
    const float ci = Qj.z * pi_, cj = ui_ * pj_;  // U_j Y_i, U_i Y_j
    float f = mj * (ci * dwi + cj * dwj + visc * dwbar) * rinv;
    a0 -= f * dx;
    a1 -= f * dy;
    a2 -= f * dz;
    du += mj * (ci * dwi + 0.5f * visc * dwbar) * w;
}

// FL lanes per particle: a lane takes every FL-th pair and the sums are
// reduced over the lanes.  A pair gathers 64 bytes of records; with one thread
// per particle the gathers of its ~70 pairs are one chain and a small set has
// too few threads to hide it.  The sums are added to the particle slots here
// rather than in a pass of their own.
template <int FL>
__global__ void __launch_bounds__(128) k_force(ForceParams p)
{
    const int i = (blockIdx.x * blockDim.x + threadIdx.x) / FL, l = threadIdx.x & (FL - 1);
    const bool valid = i < p.ng;
    const int ii = valid ? i : 0;
    const float unit = (float)p.box[4];
    const int4 Ci = p.C[ii];
    const float4 Ri = p.R[ii];
    const float4 Vi = p.V[ii];
    const float4 Qi = p.Q[ii];
    const int ci0 = Ci.x, ci1 = Ci.y, ci2 = Ci.z;
    const float ri0 = Ri.x, ri1 = Ri.y, ri2 = Ri.z;
    const float vi0 = Vi.x, vi1 = Vi.y, vi2 = Vi.z;
    const float hinv = Qi.w, rhoi = Qi.x, csi = Vi.w;
    const float pi_ = Qi.y, ui_ = Qi.z;
    float a0 = 0.f, a1 = 0.f, a2 = 0.f, du = 0.f, vs = 2.f * csi;
    if (valid) {
        const int *nb = p.nbr + (size_t)i * NGB;
        for (int k = l; k < NGB; k += FL) {
            const int j = nb[k];
            if (j == i) continue;
            pair_force(p, j, unit, ci0, ci1, ci2, ri0, ri1, ri2, vi0, vi1, vi2, hinv, pi_, ui_, rhoi, csi, a0, a1, a2,
                       du, vs);
        }
        const int b = p.roff[i], e = b + p.rcnt[i];
        for (int k = b + l; k < e; k += FL)
            pair_force(p, p.rlist[k], unit, ci0, ci1, ci2, ri0, ri1, ri2, vi0, vi1, vi2, hinv, pi_, ui_, rhoi, csi, a0,
                       a1, a2, du, vs);
    }
#pragma unroll
    for (int o = FL / 2; o > 0; o >>= 1) {
        a0 += __shfl_xor_sync(0xffffffffu, a0, o);
        a1 += __shfl_xor_sync(0xffffffffu, a1, o);
        a2 += __shfl_xor_sync(0xffffffffu, a2, o);
        du += __shfl_xor_sync(0xffffffffu, du, o);
        vs = fmaxf(vs, __shfl_xor_sync(0xffffffffu, vs, o));
    }
    if (valid && l == 0) {
        const int s = p.gslot[i];
        p.ax[s] += a0;
        p.ay[s] += a1;
        p.az[s] += a2;
        p.dudt[s] = du;
        p.vsig[i] = vs;
    }
}

// ---------------------------------------------------------------- host
static int g_knn_blocks = 0;

__global__ void __launch_bounds__(256) k_keep_support(int ng, const int *__restrict__ gslot,
                                                      const double *__restrict__ h2, double *__restrict__ s_h2)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < ng) s_h2[gslot[i]] = h2[i];
}

// The supports of a search that succeeded become the particles': they are the
// next search's starting radii and part of the saved state, so one that fails
// must not touch them (density, pressure and sound speed, which it may have
// overwritten in part, are marked invalid instead).  sph_force does the same
// on its way (k_mutual).
int sph_keep_support(gnb_ctx *c)
{
    const int ng = (int)c->n_gas;
    if (ng == 0) return GNB_OK;
    gnb::counted(k_keep_support)<<<(ng + 255) / 256, 256, 0, c->s>>>(ng, c->gslot, c->gh2, c->P[c->cur].h2);
    GNB_LAUNCH_CHECK(c, "supports");
    c->have_h = true;
    return GNB_OK;
}

int sph_density(gnb_ctx *c)
{
    int ng = (int)c->n_gas;
    if (ng == 0) return GNB_OK;
    phase_begin(c, GNB_T_HYDRO_TREE);
    PArr &a = c->P[c->cur];
    int gb = (ng + 255) / 256;
    // gas slots in Morton order (a supernova region is all gas: nothing to select)
    GasGather gg;
    gg.all = c->n_gas == c->n ? 1 : 0;
    if (!gg.all) GNB_TRY(gas_slots(c, a.type, c->n_d, c->gslot));
    gg.skey = c->skey; gg.p = a; gg.gslot = c->gslot; gg.gkey = c->gkey;
    gg.ggrank = c->ggrank; gg.C = c->fC; gg.R = c->fR;
    gg.gvx = c->gvx; gg.gvy = c->gvy; gg.gvz = c->gvz; gg.gu = c->gu; gg.gRprev = c->gRprev;
    gg.gx = c->gx; gg.gy = c->gy; gg.gz = c->gz;
    gg.ng = ng; gg.pred = c->use_pred ? 1 : 0; gg.have_h = c->have_h ? 1 : 0;
    gnb::counted(k_gas_gather)<<<gb, 256, 0, c->s>>>(gg);
    GNB_LAUNCH_CHECK(c, "gas gather");
    // hydro tree and groups of at most 32 gas particles (a lane each in the search)
    GNB_TRY(build_tree(c, c->gt, c->gkey, ng, c->ngas_d, c->cfg.n_leaf, KN_GROUP, nullptr, nullptr, nullptr, nullptr,
                       nullptr, nullptr, nullptr, nullptr, false));
    if (c->gt.nnodes >= 1 << 29) return fail(c, GNB_ECAPACITY, "hydro tree nodes");
    phase_begin(c, GNB_T_KNN);
    size_t smem = KN_WARPS * sizeof(KnnWarp);
    cudaError_t e = cudaFuncSetAttribute(k_knn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return cuda_check(c, e, "knn smem attribute");
    if (g_knn_blocks == 0) {
        int dev = 0, sms = 0, per = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_knn, KN_THREADS, smem);
        g_knn_blocks = sms * (per > 0 ? per : 1);
    }
    // particles per work item (a lane each, at most KN_GROUP).  A longer run
    // shares its walk and its candidates; a shorter one spreads a small set
    // over more warps and, in three dimensions, gathers fewer candidates per
    // member.  Measured at 30 k gas particles: 2 per item 111 us, 4 125, 8 159;
    // 1e5: 4 270, 8 300, 16 361; 210 k: 4 461, 8 453, 16 506; 1.68 M: 4 3.52
    // ms, 8 3.07, 16 2.97.
    const int steps[4] = {4, 12, 40, 256};  // gas particles per resident warp
    int sub = 1;
    for (int q : steps)
        if ((long long)ng > (long long)q * g_knn_blocks * KN_WARPS) sub *= 2;
    // work_d: [0] next item, [1] items whose radius was widened, [2] items,
    // [3] set when a particle could not be ranked
    cudaMemsetAsync(c->work_d, 0, 4 * sizeof(int), c->s);
    gnb::counted(k_knn_init)<<<304, 256, 0, c->s>>>(c->gt, sub, c->box_d, c->kR, c->kitem, c->work_d + 2);
    KnnParams p;
    p.na = c->gt.na; p.nb = c->gt.nb; p.item = c->kitem; p.kR = c->kR; p.nitems = c->work_d + 2;
    p.next = c->work_d; p.nunder = c->work_d + 1;
    p.C = c->fC; p.R = c->fR; p.ggrank = c->ggrank; p.gu = c->gu;
    p.gx = c->gx; p.gy = c->gy; p.gz = c->gz; p.box = c->box_d;
    p.rprev = c->gRprev;
    p.margin = c->knn_margin;
    p.failed = c->work_d + 3;
    p.nbr = c->nbr; p.nd2 = c->nd2; p.h2 = c->gh2; p.h2b = c->gh2b; p.h = c->gh; p.E = c->gE; p.g64 = c->g64;
    p.gvx = c->gvx; p.gvy = c->gvy; p.gvz = c->gvz; p.V = c->fV; p.Q = c->fQ;
    p.gslot = c->gslot; p.s_rho = c->rho; p.s_pres = c->pres; p.s_cs = c->cs;
    p.gamma = (float)c->cfg.gamma; p.pressure = c->cfg.sph_variant;
    c->density_valid = c->nbr_valid = false;  // overwritten from here on
    gnb::counted(k_knn)<<<g_knn_blocks, KN_THREADS, smem, c->s>>>(p);
    GNB_LAUNCH_CHECK(c, "knn");
    cudaMemcpyAsync(c->pinned_i, c->work_d, 4 * sizeof(int), cudaMemcpyDeviceToHost, c->s);
    GNB_TRY(cuda_check(c, cudaStreamSynchronize(c->s), "knn sync"));
    if (c->pinned_i[3]) return fail(c, GNB_ECAPACITY, "kNN selection buffer overflow");
    c->stats[GNB_S_KNN_PASSES] = 1;
    // the next evaluation's margin: wider when more than 4 % of the items
    // needed a larger radius, narrower (to 1.01) below 1 %
    if (c->have_h) {
        const double under = (double)c->pinned_i[1] / (double)std::max(1, c->pinned_i[2]);
        if (under > 0.04) c->knn_margin = std::min(1.5f, c->knn_margin * 1.05f);
        else if (under < 0.01) c->knn_margin = std::max(1.01f, c->knn_margin / 1.02f);
    }
    c->stats[GNB_S_GAS_NODES] = c->gt.nnodes;
    phase_end(c);
    c->nbr_valid = true;
    return GNB_OK;
}

int sph_force(gnb_ctx *c)
{
    int ng = (int)c->n_gas;
    if (ng == 0) return GNB_OK;
    phase_begin(c, GNB_T_FORCE);
    // lanes per particle: more spread a small set over the chip, fewer do less
    // reduction and bit bookkeeping.  Phase time, lists + force, one thread per
    // particle -> 16 and 8 lanes -> 8 and 4: 4,096 gas particles 164 -> 37 ->
    // 47 us, 1e5 242 -> 135 -> 137, 210 k 424 -> 259 -> 243, 1.68 M 2464 -> 1943
    // -> 1733.
    const bool few = ng < 150000;
    const int sl = few ? 16 : 8, fl = few ? 8 : 4;
    const int gb = (ng + 255) / 256, gbl = (int)(((long long)ng * sl + 255) / 256);
    cudaMemsetAsync(c->rcnt, 0, sizeof(int) * ng, c->s);
    gnb::counted(few ? k_mutual<16> : k_mutual<8>)<<<gbl, 256, 0, c->s>>>(
        ng, c->nbr, c->nd2, c->gE, c->gh2, c->gh2b, c->g64, c->ggrank, c->gx, c->gy, c->gz, c->mut, c->rcnt, c->rtot_d,
        c->gslot, c->P[c->cur].h2);
    c->have_h = true;
    gnb::counted(k_rev_off)<<<gb, 256, 0, c->s>>>(ng, c->rcnt, c->roff, c->rcur, c->rtot_d);
    gnb::counted(few ? k_rev_fill<16> : k_rev_fill<8>)<<<gbl, 256, 0, c->s>>>(ng, c->nbr, c->mut, c->rcur, c->rlist);
    GNB_LAUNCH_CHECK(c, "symmetric lists");
    ForceParams p;
    p.ng = ng; p.nbr = c->nbr; p.roff = c->roff; p.rcnt = c->rcnt; p.rlist = c->rlist;
    p.C = c->fC; p.R = c->fR; p.V = c->fV; p.Q = c->fQ;
    p.box = c->box_d; p.alpha = (float)c->cfg.alpha_visc;
    p.gslot = c->gslot;
    p.ax = c->ax; p.ay = c->ay; p.az = c->az; p.dudt = c->dudt; p.vsig = c->gvsig;
    gnb::counted(few ? k_force<8> : k_force<4>)<<<(int)(((long long)ng * fl + 127) / 128), 128, 0, c->s>>>(p);
    GNB_LAUNCH_CHECK(c, "sph force");
    phase_end(c);
    return GNB_OK;
}

}  // namespace gnb
