// sort.cu -- root box, Morton keys and the space-filling-curve sort
// (tree construction, Sec. 3.4 and 5.2.2 of Hirashima et al., SC'25).
//
// Root box: lo_k = min x_k, ext = max_k(max x_k - lo_k), L = 2^ceil(log2 ext)
// (L = 1 when ext = 0), unit = L / 2^21.  Cell c_k = min(floor((x_k - lo_k) *
// 2^21 / L), 2^21 - 1) with the FP64-rounded difference; the key interleaves bit b
// of c_x, c_y, c_z at 3b+2, 3b+1, 3b.  Particles are ordered by (key, caller
// index): a stable LSD radix sort of the keys in their current slot order by
// the top 48 bits, then the short runs that agree there put in (key, caller
// index) order (see the ties section).
#include <algorithm>
#include <utility>

#include "common.cuh"
#include "morton.cuh"

namespace gnb {

// ---------------------------------------------------------------- root box
// Min/max words accumulated by all blocks; the last block to finish (a ticket
// counter, no waiting) forms box = {lo_x, lo_y, lo_z, L, unit} and puts the
// words and the counter back to their start values for the next call.
__global__ void k_mm_init(unsigned long long *mm)
{
    minmax_init(mm, threadIdx.x);
    if (threadIdx.x == 7) mm[7] = 0ull;  // blocks done
}

__global__ void __launch_bounds__(256) k_root_box(const double *__restrict__ x, const double *__restrict__ y,
                                                  const double *__restrict__ z, int n, unsigned long long *mm,
                                                  double *box, int *status)
{
    __shared__ bool last;
    minmax_accumulate(x, y, z, n, mm);
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        last = atomicAdd(&mm[7], 1ull) == gridDim.x - 1;
        __threadfence();
    }
    __syncthreads();
    if (!last) return;
    if (threadIdx.x == 0) {
        unsigned long long w[7];
        for (int k = 0; k < 7; k++) w[k] = *(volatile unsigned long long *)&mm[k];
        if (box_from_minmax(w, box)) atomicOr(status, ST_BAD_INPUT);
    }
    __syncthreads();
    if (threadIdx.x < 7) minmax_init(mm, threadIdx.x);
    if (threadIdx.x == 7) mm[7] = 0ull;
}

int root_box(gnb_ctx *c)
{
    int n = (int)c->n;
    if (!c->mm_ready) {
        gnb::counted(k_mm_init)<<<1, 32, 0, c->s>>>(c->mm_d);
        c->mm_ready = true;
    }
    int blocks = (n + 255) / 256;
    if (blocks > 1216) blocks = 1216;
    gnb::counted(k_root_box)<<<blocks, 256, 0, c->s>>>(c->P[c->cur].x, c->P[c->cur].y, c->P[c->cur].z, n, c->mm_d,
                                                      c->box_d, c->status_d);
    GNB_LAUNCH_CHECK(c, "root box");
    return GNB_OK;
}

#define TIE_SHIFT 16  // key bits below the sorted ones (see the ties section)
#define TIE_FIRST_DIGIT (TIE_SHIFT / 8)

// A warp's digits F .. 7 of its keys into the block's histograms.  Near-sorted
// keys share their high digits: one addition where the warp agrees instead
// of 32 to one word.
template <int F>
__device__ __forceinline__ void digit_count(int (*h)[256], uint64_t k, bool valid)
{
    const unsigned vb = __ballot_sync(0xffffffffu, valid);
    if (vb == 0u) return;
    const int lead = __ffs(vb) - 1;
#pragma unroll
    for (int q = F; q < 8; q++) {
        const int d = (int)(k >> (8 * q)) & 255;
        const int d0 = __shfl_sync(0xffffffffu, d, lead);
        if (__all_sync(0xffffffffu, !valid || d == d0)) {
            if ((threadIdx.x & 31) == lead) atomicAdd(&h[q - F][d], __popc(vb));
        } else if (valid) {
            atomicAdd(&h[q - F][d], 1);
        }
    }
}

// ---------------------------------------------------------------- Morton
// Keys scattered to caller order, for the whole-key sort that a long run of
// equal 48-bit prefixes needs (see morton_and_sort).
__global__ void k_morton(PArr p, int n, const double *__restrict__ box, uint64_t *__restrict__ keyo,
                         int *__restrict__ valo, int *__restrict__ slot_of_orig)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int lexp = box_lexp(box[3]);
    const uint64_t k = morton_key(grid_cell(p.x[i], box[0], lexp), grid_cell(p.y[i], box[1], lexp),
                                  grid_cell(p.z[i], box[2], lexp));
    int o = p.orig[i];
    keyo[o] = k;
    valo[o] = o;
    slot_of_orig[o] = i;
}

// Key of every slot (the first sorting pass pairs it with the slot itself;
// ties are put into caller order afterwards, see k_tie_fix), the FP32
// remainder of each coordinate within its grid cell (res: three arrays of n,
// slot order) for the permutation, and the histograms of the digits to be
// sorted (hist[8][256], see the radix sort).
__global__ void __launch_bounds__(256) k_keys(const double *__restrict__ x, const double *__restrict__ y,
                                              const double *__restrict__ z, int n, const double *__restrict__ box,
                                              uint64_t *__restrict__ key, float *__restrict__ res,
                                              int *__restrict__ hist)
{
    __shared__ int h[8 - TIE_FIRST_DIGIT][256];
    for (int k = threadIdx.x; k < (8 - TIE_FIRST_DIGIT) * 256; k += blockDim.x) (&h[0][0])[k] = 0;
    __syncthreads();
    const int lexp = box_lexp(box[3]);
    for (int b = blockIdx.x * blockDim.x; b < n; b += gridDim.x * blockDim.x) {
        const int i = b + threadIdx.x;
        const bool valid = i < n;
        uint64_t k = 0;
        if (valid) {
            float r0, r1, r2;
            const int c0 = grid_cell(x[i], box[0], lexp, &r0);
            const int c1 = grid_cell(y[i], box[1], lexp, &r1);
            const int c2 = grid_cell(z[i], box[2], lexp, &r2);
            k = morton_key(c0, c1, c2);
            key[i] = k;
            res[i] = r0;
            res[(size_t)n + i] = r1;
            res[2 * (size_t)n + i] = r2;
        }
        digit_count<TIE_FIRST_DIGIT>(h, k, valid);
    }
    __syncthreads();
    for (int k = threadIdx.x; k < (8 - TIE_FIRST_DIGIT) * 256; k += blockDim.x)
        if ((&h[0][0])[k]) atomicAdd(&hist[TIE_FIRST_DIGIT * 256 + k], (&h[0][0])[k]);
}

// ---------------------------------------------------------------- ties
// The slot-order sort runs over the top 48 key bits only (levels 1 to 16),
// stably, so pairs whose keys agree there are left in old-slot order; the
// order wanted is (key, caller index).  Such runs are particles in the same
// level-16 cell (a 2^-16 part of the box side), a few at most in any real
// set: one thread per run puts it in order by insertion sort, for runs of at
// most TIE_MAX entries.  st[0] = 1 when some run exists, st[1] = the longest
// (capped at TIE_MAX + 1); a longer run is left to the caller-order sort.
#define TIE_MAX 4096

__device__ __forceinline__ bool tie(uint64_t a, uint64_t b) { return (a >> TIE_SHIFT) == (b >> TIE_SHIFT); }

__global__ void k_tie_detect(const uint64_t *__restrict__ k, int n, int *__restrict__ st)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i + 1 >= n || !tie(k[i], k[i + 1])) return;
    if (i > 0 && tie(k[i - 1], k[i])) return;  // not the run's start
    int e = i + 1;
    while (e < n && e - i <= TIE_MAX && tie(k[e], k[i])) e++;
    atomicOr(&st[0], 1);
    atomicMax(&st[1], e - i);
}

__global__ void k_tie_fix(uint64_t *__restrict__ k, int n, int *__restrict__ val, const int *__restrict__ orig)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i + 1 >= n || !tie(k[i], k[i + 1])) return;
    if (i > 0 && tie(k[i - 1], k[i])) return;
    int e = i + 1;
    while (e < n && tie(k[e], k[i])) e++;
    for (int a = i + 1; a < e; a++) {  // insertion sort of the pairs [i, e) by (key, orig[val])
        const uint64_t kv = k[a];
        const int v = val[a], ov = orig[v];
        int b = a - 1;
        while (b >= i && (k[b] > kv || (k[b] == kv && orig[val[b]] > ov))) {
            k[b + 1] = k[b];
            val[b + 1] = val[b];
            b--;
        }
        k[b + 1] = kv;
        val[b + 1] = v;
    }
}

// ---------------------------------------------------------------- radix sort
// Stable LSD radix sort of (64-bit key, 32-bit value), 8 bits per pass, one
// kernel per pass: the digit histograms of all passes are counted once, up
// front (they do not depend on the order; those of the Morton keys come with
// the keys), and a tile finds where its run of each digit starts from the
// counts that the tiles before it publish.  The scheme is the single-pass scan
// with decoupled look-back of Merrill and Garland (NVIDIA technical report
// NVR-2016-002), applied to every digit as in the one-sweep radix sort of
// Adinets and Merrill (arXiv 2206.01784).  A tile takes its number from a
// ticket counter, so every tile it waits for is already running.
//
// A tile's pairs are first sorted by digit in shared memory, stably, then
// written out in that order, so consecutive threads write consecutive
// addresses of each digit's run instead of one scattered store each.  Each
// warp ranks its own contiguous ITEMS * 32 pairs of the tile (rounds of 32 in
// order, lanes in order within a round) against per-warp digit counters, with
// warp synchronisation only; one block-wide step then turns the counters into
// each warp's offset within the digit's run of the tile.
#define RS_THREADS 256
#define RS_BATCH 8            // published counts read at once in the look-back
#define RS_AGG (1u << 30)     // the tile's own count of the digit
#define RS_PRE (2u << 30)     // the count of the digit in this tile and all before it
#define RS_SPINS (1 << 20)    // look-back reads without progress before giving up
#define RS_DEAD (1 << 30)     // in a pass's ticket counter: an earlier pass gave up

struct RsState {
    int *hist;        // [8][256] digit histograms
    int *ticket;      // [8] tiles started per pass
    unsigned *state;  // [passes][ntiles][256] published counts
    int *flag;        // set when a look-back gave up
};

template <int ITEMS>
struct RsSmem {
    uint64_t k[RS_THREADS * ITEMS];
    int v[RS_THREADS * ITEMS];
    int wc[RS_THREADS / 32][256];  // per-warp digit counts, then each warp's offset in the digit's run
    int lstart[256];               // first local position of each digit
    int goff[256];                 // global position of each digit's first pair of this tile
    int ws[RS_THREADS / 32], wh[RS_THREADS / 32];
    int tile, stop;
};

__device__ __forceinline__ unsigned ld_relaxed(const unsigned *p)
{
    unsigned v;
    asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void st_relaxed(unsigned *p, unsigned v)
{
    asm volatile("st.relaxed.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// Lanes whose low eight bits of d equal this lane's, among the valid ones: eight
// ballots.
__device__ __forceinline__ unsigned digit_peers(unsigned d, bool valid)
{
    unsigned p = __ballot_sync(0xffffffffu, valid);
#pragma unroll
    for (int b = 0; b < 8; b++) {
        const unsigned m = __ballot_sync(0xffffffffu, (d >> b) & 1u);
        p &= (d >> b) & 1u ? m : ~m;
    }
    return valid ? p : 1u << (threadIdx.x & 31);
}

// FIRST: the values are the slots themselves (vin is not read)
template <int ITEMS, bool FIRST>
__global__ void __launch_bounds__(RS_THREADS, 3) k_rs_pass(const uint64_t *__restrict__ kin,
                                                          const int *__restrict__ vin, uint64_t *__restrict__ kout,
                                                          int *__restrict__ vout, int n, int shift,
                                                          const int *__restrict__ hist, int *ticket, unsigned *state,
                                                          int *flag)
{
    extern __shared__ __align__(16) unsigned char rs_raw[];
    RsSmem<ITEMS> &S = *reinterpret_cast<RsSmem<ITEMS> *>(rs_raw);
    constexpr int TILE = RS_THREADS * ITEMS;
    const int t = threadIdx.x, w = t >> 5, lane = t & 31;
    const unsigned lt = (1u << lane) - 1u;
    if (t == 0) {
        S.tile = atomicAdd(ticket, 1);
        S.stop = 0;
    }
#pragma unroll
    for (int q = 0; q < RS_THREADS / 32; q++) S.wc[q][t] = 0;
    const int hd = hist[t];
    __syncthreads();
    const int tile = S.tile;
    // an earlier pass that gave up left places unwritten: its output no longer
    // has the digits that were counted, and their positions could lie beyond
    // the arrays
    if (tile >= RS_DEAD) return;
    const int base = tile * TILE;
    const int cnt = min(TILE, n - base);
    uint64_t key[ITEMS];
    int lr[ITEMS];
#pragma unroll
    for (int r = 0; r < ITEMS; r++) {
        const int i = w * (ITEMS * 32) + r * 32 + lane;
        key[r] = i < cnt ? kin[base + i] : 0ull;
    }
    // ranks, up to eight rounds at a time: the lanes of equal digit of each
    // round first, then one counter addition per digit and round by its first
    // lane (in round order; the old values are only used after the last of
    // them, so the additions overlap), then every lane's rank from its
    // leader's old value.  (With a match instruction, a read, a write and an
    // exchange per round, one after the other, those latencies set the time: a
    // pass over 6.4 M pairs 80 us, cold cache, now 64.)
    constexpr int GR = ITEMS < 8 ? ITEMS : 8;
#pragma unroll
    for (int g = 0; g < ITEMS; g += GR) {
        unsigned peers[GR];
#pragma unroll
        for (int q = 0; q < GR; q++) {
            const int r = g + q, i = w * (ITEMS * 32) + r * 32 + lane;
            peers[q] = digit_peers((unsigned)(key[r] >> shift), i < cnt);
        }
#pragma unroll
        for (int q = 0; q < GR; q++) {
            const int r = g + q, i = w * (ITEMS * 32) + r * 32 + lane;
            lr[r] = 0;
            if (i < cnt && (peers[q] & lt) == 0u)
                lr[r] = atomicAdd(&S.wc[w][(key[r] >> shift) & 255u], __popc(peers[q]));
            __syncwarp();
        }
#pragma unroll
        for (int q = 0; q < GR; q++)
            lr[g + q] = __shfl_sync(0xffffffffu, lr[g + q], __ffs(peers[q]) - 1) + __popc(peers[q] & lt);
    }
    __syncthreads();
    // digit t: offsets of the warps within the digit's run; publish the count
    int run = 0;
#pragma unroll
    for (int q = 0; q < RS_THREADS / 32; q++) {
        const int c = S.wc[q][t];
        S.wc[q][t] = run;
        run += c;
    }
    unsigned *mine = state + (size_t)tile * 256 + t;
    st_relaxed(mine, (tile == 0 ? RS_PRE : RS_AGG) | (unsigned)run);
    // exclusive scans over the 256 digits: of the tile's counts and of all counts
    int gbase;
    {
        int x = run, y = hd;
        for (int o = 1; o < 32; o <<= 1) {
            const int a = __shfl_up_sync(0xffffffffu, x, o), b = __shfl_up_sync(0xffffffffu, y, o);
            if (lane >= o) { x += a; y += b; }
        }
        if (lane == 31) { S.ws[w] = x; S.wh[w] = y; }
        __syncthreads();
        int px = 0, py = 0;
        for (int q = 0; q < w; q++) { px += S.ws[q]; py += S.wh[q]; }
        S.lstart[t] = px + x - run;
        gbase = py + y - hd;
    }
    int val[ITEMS];  // (read here: they would hold registers through the ranking)
#pragma unroll
    for (int r = 0; r < ITEMS; r++) {
        const int i = w * (ITEMS * 32) + r * 32 + lane;
        val[r] = FIRST ? base + i : (i < cnt ? vin[base + i] : 0);
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < ITEMS; r++) {
        const int i = w * (ITEMS * 32) + r * 32 + lane;
        if (i < cnt) {
            const int d = (int)((key[r] >> shift) & 255u);
            const int lp = S.lstart[d] + S.wc[w][d] + lr[r];
            S.k[lp] = key[r];
            S.v[lp] = val[r];
        }
    }
    // look-back: the digit's count in the tiles before this one
    int before = 0;
    for (int p = tile - 1, spins = 0; p >= 0;) {
        unsigned s[RS_BATCH];
#pragma unroll
        for (int q = 0; q < RS_BATCH; q++) s[q] = ld_relaxed(state + (size_t)max(p - q, 0) * 256 + t);
        bool moved = false;
#pragma unroll
        for (int q = 0; q < RS_BATCH; q++) {
            if (p < 0 || s[q] < RS_AGG) break;  // past the first tile, or not published yet
            before += (int)(s[q] & (RS_AGG - 1u));
            p = s[q] >= RS_PRE ? -1 : p - 1;
            moved = true;
        }
        if (moved) spins = 0;
        else if (++spins > RS_SPINS) {  // cannot happen unless a block was lost
            S.stop = 1;
            atomicOr(flag, 1);
            for (int q = (shift >> 3) + 1; q < 8; q++) atomicOr(ticket + q - (shift >> 3), RS_DEAD);
            break;
        }
    }
    if (tile > 0) st_relaxed(mine, RS_PRE | (unsigned)(before + run));
    S.goff[t] = gbase + before;
    __syncthreads();
    if (S.stop) return;
    for (int pos = t; pos < cnt; pos += RS_THREADS) {
        const uint64_t k = S.k[pos];
        const int d = (int)((k >> shift) & 255u);
        const int dst = S.goff[d] + pos - S.lstart[d];
        kout[dst] = k;
        vout[dst] = S.v[pos];
    }
}

// Histograms of all digits from digit F up (the Morton keys' come with the keys).
template <int F>
__global__ void __launch_bounds__(256) k_rs_hist(const uint64_t *__restrict__ key, int n, int *__restrict__ hist)
{
    __shared__ int h[8 - F][256];
    for (int k = threadIdx.x; k < (8 - F) * 256; k += blockDim.x) (&h[0][0])[k] = 0;
    __syncthreads();
    for (int b = blockIdx.x * blockDim.x; b < n; b += gridDim.x * blockDim.x) {
        const int i = b + threadIdx.x;
        digit_count<F>(h, i < n ? key[i] : 0ull, i < n);
    }
    __syncthreads();
    for (int k = threadIdx.x; k < (8 - F) * 256; k += blockDim.x)
        if ((&h[0][0])[k]) atomicAdd(&hist[F * 256 + k], (&h[0][0])[k]);
}

// Pairs per thread of a tile.  Small tiles spread a small set over the chip and
// shorten the serial ranking rounds; large ones write longer runs and have
// fewer predecessors to look back to.  Sort phase with 4 / 8 / 16: 8,192
// particles 75 / 85 / - us, 150,001 118 / 126 / 139, 300,007 177 / 172 / 184,
// 2^20 - / 276 / 254 (histogram, scan and scatter kernels per pass: 186, 217,
// 324 and 330).
static int rs_items(int n) { return n <= 200000 ? 4 : (n <= 500000 ? 8 : 16); }

// Words of a sort of n pairs: histograms, tickets, the give-up flag and the
// published counts of eight passes.
static size_t rs_words(int n)
{
    const int tile = RS_THREADS * rs_items(n);
    return 8 * 256 + 16 + 8 * (size_t)((n + tile - 1) / tile) * 256;
}

// Scratch for sorts of up to n pairs (smaller tiles below the lines of
// rs_items): allocated with the particles, about 8 bytes each.
int sort_reserve(gnb_ctx *c, int n)
{
    const size_t words = std::max({rs_words(n), rs_words(std::min(n, 200000)), rs_words(std::min(n, 500000))});
    if (c->rs_words >= words) return GNB_OK;
    drop(c, c->rs_buf);
    c->rs_words = 0;
    GNB_TRY(dalloc(c, &c->rs_buf, words));
    c->rs_words = words;
    return GNB_OK;
}

// The scratch of a sort of n pairs, cleared.
static int rs_begin(gnb_ctx *c, int n, RsState *st)
{
    const size_t words = rs_words(n);
    GNB_TRY(sort_reserve(c, n));
    st->hist = c->rs_buf;
    st->ticket = c->rs_buf + 8 * 256;
    st->flag = c->rs_buf + 8 * 256 + 8;
    st->state = (unsigned *)(c->rs_buf + 8 * 256 + 16);
    GNB_TRY(cuda_check(c, cudaMemsetAsync(c->rs_buf, 0, words * sizeof(int), c->s), "radix sort scratch"));
    if (c->sort_gives_up >= 0) {  // (set by tests)
        const int later = c->sort_gives_up + 1;
        c->sort_gives_up = -1;
        GNB_TRY(cuda_check(c, cudaMemsetAsync(st->flag, 1, 1, c->s), "radix sort flag"));
        GNB_TRY(cuda_check(c, cudaMemsetAsync(st->ticket + later, RS_DEAD >> 24, (8 - later) * sizeof(int), c->s),
                           "radix sort flag"));
    }
    return GNB_OK;
}

template <int ITEMS, bool FIRST>
static int rs_pass(gnb_ctx *c, const RsState &st, const uint64_t *kin, const int *vin, uint64_t *kout, int *vout, int n,
                   int pass)
{
    // a tile needs more than the default 48 KB of shared memory
    const cudaError_t e = cudaFuncSetAttribute(k_rs_pass<ITEMS, FIRST>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                               (int)sizeof(RsSmem<ITEMS>));
    if (e != cudaSuccess) return cuda_check(c, e, "radix sort shared memory attribute");
    const int ntiles = (n + RS_THREADS * ITEMS - 1) / (RS_THREADS * ITEMS);
    gnb::counted(k_rs_pass<ITEMS, FIRST>)<<<ntiles, RS_THREADS, sizeof(RsSmem<ITEMS>), c->s>>>(
        kin, vin, kout, vout, n, 8 * pass, st.hist + 256 * pass, st.ticket + pass,
        st.state + (size_t)pass * ntiles * 256, st.flag);
    return GNB_OK;
}

// The passes from digit `first` up over (k0, v0) with (k1, v1) as the
// ping-pong buffers, histograms counted; 8 - first is even, so the sorted
// pairs end in (k0, v0).  slots: the values are the slots 0 .. n - 1 (v0 is
// not read).
static int rs_passes(gnb_ctx *c, const RsState &st, uint64_t *k0, int *v0, uint64_t *k1, int *v1, int n, int first,
                     bool slots)
{
    for (int pass = first; pass < 8; pass++) {
        const bool odd = (pass - first) & 1, f = slots && pass == first;
        const uint64_t *ki = odd ? k1 : k0;
        const int *vi = odd ? v1 : v0;
        uint64_t *ko = odd ? k0 : k1;
        int *vo = odd ? v0 : v1;
        switch (rs_items(n)) {
        case 4: GNB_TRY(f ? (rs_pass<4, true>(c, st, ki, vi, ko, vo, n, pass))
                          : (rs_pass<4, false>(c, st, ki, vi, ko, vo, n, pass))); break;
        case 8: GNB_TRY(f ? (rs_pass<8, true>(c, st, ki, vi, ko, vo, n, pass))
                          : (rs_pass<8, false>(c, st, ki, vi, ko, vo, n, pass))); break;
        default: GNB_TRY(f ? (rs_pass<16, true>(c, st, ki, vi, ko, vo, n, pass))
                           : (rs_pass<16, false>(c, st, ki, vi, ko, vo, n, pass))); break;
        }
    }
    GNB_LAUNCH_CHECK(c, "radix sort");
    return GNB_OK;
}

static int rs_gave_up(gnb_ctx *c) { return fail(c, GNB_ETIMEOUT, "a bounded wait in the radix sort ran out"); }

// Stable sort of n (64-bit key, 32-bit value) pairs held in (k0, v0) by the
// whole key, with (k1, v1) as the ping-pong buffers; the sorted pairs end in
// (k0, v0).  Waits for the result.
int radix_sort_pairs(gnb_ctx *c, uint64_t *k0, int *v0, uint64_t *k1, int *v1, int n)
{
    RsState st;
    GNB_TRY(rs_begin(c, n, &st));
    gnb::counted(k_rs_hist<0>)<<<std::min((n + 1023) / 1024, 1216), 256, 0, c->s>>>(k0, n, st.hist);
    GNB_TRY(rs_passes(c, st, k0, v0, k1, v1, n, 0, false));
    GNB_TRY(cuda_check(c, cudaMemcpyAsync(c->pinned_i + 60, st.flag, sizeof(int), cudaMemcpyDeviceToHost, c->s),
                       "radix sort flag"));
    GNB_TRY(cuda_check(c, cudaStreamSynchronize(c->s), "radix sort sync"));
    return c->pinned_i[60] ? rs_gave_up(c) : GNB_OK;
}

// ---------------------------------------------------------------- permute
// New slot i takes old slot src[i] = slot_of_orig[sorted caller index].
__global__ void k_src(const int *__restrict__ sval, const int *__restrict__ slot_of_orig,
                      int *__restrict__ src, int n)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) src[i] = slot_of_orig[sval[i]];
}

// New slot i takes old slot src[i]; its grid cell comes from its sorted key
// and its remainder within the cell from the key pass (res, old-slot order).
__global__ void k_permute(PArr a, PArr b, const int *__restrict__ src, int n, const uint64_t *__restrict__ skey,
                          const float *__restrict__ res)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    int s = src[i];
    b.x[i] = a.x[s]; b.y[i] = a.y[s]; b.z[i] = a.z[s]; b.h2[i] = a.h2[s]; b.id[i] = a.id[s];
    b.vx[i] = a.vx[s]; b.vy[i] = a.vy[s]; b.vz[i] = a.vz[s];
    b.m[i] = a.m[s]; b.eps[i] = a.eps[s]; b.u[i] = a.u[s];
    b.vpx[i] = a.vpx[s]; b.vpy[i] = a.vpy[s]; b.vpz[i] = a.vpz[s]; b.up[i] = a.up[s];
    b.orig[i] = a.orig[s]; b.grank[i] = a.grank[s];
    b.type[i] = a.type[s];
    const uint64_t k = skey[i];
    b.cx[i] = compact3(k >> 2);
    b.cy[i] = compact3(k >> 1);
    b.cz[i] = compact3(k);
    b.rx[i] = res[s];
    b.ry[i] = res[(size_t)n + s];
    b.rz[i] = res[2 * (size_t)n + s];
}

// The first sort after an upload starts from the caller's order, so its
// gather sources are spread over whole arrays: one pass per array keeps that
// array (at most 8 bytes a particle) in L2 while it is gathered, instead of
// one pass whose 22 sources together are far larger than L2 (on the 2^24
// disk the single pass took 7.1 ms against 0.73 ms for the near-sorted
// permutations of later steps).  Up to PERM_ONE_PASS particles all sources fit
// in L2 together (about 150 bytes a particle) and 22 launches cost more than
// the single pass.
#define PERM_ONE_PASS 500000
template <class T>
__global__ void k_gather1(const T *__restrict__ a, T *__restrict__ b, const int *__restrict__ src, int n)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) b[i] = a[src[i]];
}

__global__ void k_cells_of_key(const uint64_t *__restrict__ skey, int n, int *__restrict__ cx, int *__restrict__ cy,
                               int *__restrict__ cz)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const uint64_t k = skey[i];
    cx[i] = compact3(k >> 2);
    cy[i] = compact3(k >> 1);
    cz[i] = compact3(k);
}

template <class T>
static void gather1(gnb_ctx *c, const T *a, T *b, const int *src, int n)
{
    gnb::counted(k_gather1<T>)<<<(n + 255) / 256, 256, 0, c->s>>>(a, b, src, n);
}

static int permute_per_array(gnb_ctx *c, const PArr &a, PArr &b, const int *src, int n)
{
    for (auto q : {std::make_pair(a.x, b.x), std::make_pair(a.y, b.y), std::make_pair(a.z, b.z),
                   std::make_pair(a.h2, b.h2)})
        gather1<double>(c, q.first, q.second, src, n);
    gather1<int64_t>(c, a.id, b.id, src, n);
    for (auto q : {std::make_pair(a.vx, b.vx), std::make_pair(a.vy, b.vy), std::make_pair(a.vz, b.vz),
                   std::make_pair(a.m, b.m), std::make_pair(a.eps, b.eps), std::make_pair(a.u, b.u),
                   std::make_pair(a.vpx, b.vpx), std::make_pair(a.vpy, b.vpy), std::make_pair(a.vpz, b.vpz),
                   std::make_pair(a.up, b.up)})
        gather1<float>(c, q.first, q.second, src, n);
    const float *res = c->kres;
    gather1<float>(c, res, b.rx, src, n);
    gather1<float>(c, res + (size_t)n, b.ry, src, n);
    gather1<float>(c, res + 2 * (size_t)n, b.rz, src, n);
    gather1<int>(c, a.orig, b.orig, src, n);
    gather1<int>(c, a.grank, b.grank, src, n);
    gather1<uint8_t>(c, a.type, b.type, src, n);
    gnb::counted(k_cells_of_key)<<<(n + 255) / 256, 256, 0, c->s>>>(c->skey, n, b.cx, b.cy, b.cz);
    GNB_LAUNCH_CHECK(c, "permute per array");
    return GNB_OK;
}

int morton_and_sort(gnb_ctx *c)
{
    int n = (int)c->n;
    GNB_TRY(root_box(c));
    int nb = (n + 255) / 256;
    PArr &a = c->P[c->cur];
    // keys in slot order (the particles are near their previous Morton
    // order), stable sort by the top 48 bits, then runs into (key, caller
    // index) order
    RsState st;
    GNB_TRY(rs_begin(c, n, &st));
    gnb::counted(k_keys)<<<std::min(nb, 1216), 256, 0, c->s>>>(a.x, a.y, a.z, n, c->box_d, c->skey, c->kres, st.hist);
    GNB_LAUNCH_CHECK(c, "keys");
    GNB_TRY(rs_passes(c, st, c->skey, c->sval, c->skey2, c->sval2, n, TIE_FIRST_DIGIT, true));
    gnb::counted(k_tie_detect)<<<nb, 256, 0, c->s>>>(c->skey, n, st.flag + 1);
    GNB_LAUNCH_CHECK(c, "tie detect");
    GNB_TRY(cuda_check(c, cudaMemcpyAsync(c->pinned_i + 60, st.flag, 3 * sizeof(int), cudaMemcpyDeviceToHost, c->s),
                       "tie flag"));
    GNB_TRY(cuda_check(c, cudaStreamSynchronize(c->s), "tie flag sync"));
    const int *flags = c->pinned_i + 60;  // {look-back gave up, some run of ties, the longest}
    if (flags[0]) return rs_gave_up(c);
    if (flags[1] && flags[2] <= TIE_MAX) {
        gnb::counted(k_tie_fix)<<<nb, 256, 0, c->s>>>(c->skey, n, c->sval, a.orig);
        GNB_LAUNCH_CHECK(c, "tie fix");
        std::swap(c->src, c->sval);
    } else if (flags[1]) {
        // a run of more than TIE_MAX: sort by the whole key in caller order
        // (keys scattered to the caller index, stable sort, slot map)
        gnb::counted(k_morton)<<<nb, 256, 0, c->s>>>(a, n, c->box_d, c->skey, c->sval, c->slot_of_orig);
        GNB_LAUNCH_CHECK(c, "morton");
        GNB_TRY(radix_sort_pairs(c, c->skey, c->sval, c->skey2, c->sval2, n));
        gnb::counted(k_src)<<<nb, 256, 0, c->s>>>(c->sval, c->slot_of_orig, c->src, n);
    } else {
        std::swap(c->src, c->sval);  // the old slot of each sorted particle
    }
    PArr &b = c->P[1 - c->cur];
    if (c->slots_caller && n > PERM_ONE_PASS) {
        GNB_TRY(permute_per_array(c, a, b, c->src, n));
    } else {
        gnb::counted(k_permute)<<<nb, 256, 0, c->s>>>(a, b, c->src, n, c->skey, c->kres);
        GNB_LAUNCH_CHECK(c, "permute");
    }
    c->slots_caller = false;
    c->cur = 1 - c->cur;
    if (c->hier_on) GNB_TRY(hier_permute(c));  // per-particle step state follows the particles
    return GNB_OK;
}

}  // namespace gnb
