// Morton octree build and dual-tree interaction lists on the GPU.
//
// Sec. 2.1 of Yokota & Barba (arXiv:1106.2176) subdivides space hierarchically
// into near and far regions; Sec. 2.2 and Sec. 5 index the boxes by a Morton
// key at a prescribed maximum level and address particles through sorted
// indices with start/offset ranges. This file builds exactly that, all on the
// device and integer or correctly rounded FP64, so that keys, permutation,
// cells and lists are bit-identical to an independent CPU implementation:
//   bounding cube -> 21-bit quantisation -> 63-bit Morton keys -> stable LSD
//   radix sort -> top-down cell split (ncrit) -> level-synchronous dual
//   traversal with the theta MAC -> CSR lists.
// Same-level M2L pairs are not stored: two existing cells of one level form an
// M2L pair exactly when their lattice offset lies in the stencil of the
// target's octant (the MAC accepts them and rejects their parents), so the M2L
// kernels enumerate them through a per-level lattice lookup.
#include <algorithm>
#include <climits>
#include <cmath>

#include "fmm_internal.cuh"

namespace fmm {

// ---------------------------------------------------------------------------
// small helpers
// ---------------------------------------------------------------------------
static inline unsigned nblocks(int64_t n, int bs) { return (unsigned)((n + bs - 1) / bs); }

void check_launch(const char *what)
{
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) throw Error{FMM_ECUDA, std::string(what) + ": " + cudaGetErrorString(e)};
}

__device__ __forceinline__ unsigned long long ord_enc(double d)
{
    unsigned long long u = (unsigned long long)__double_as_longlong(d);
    return (u >> 63) ? ~u : (u | 0x8000000000000000ull);
}

__device__ __forceinline__ double ord_dec(unsigned long long e)
{
    unsigned long long u = (e >> 63) ? (e & 0x7fffffffffffffffull) : ~e;
    return __longlong_as_double((long long)u);
}

// ---------------------------------------------------------------------------
// exclusive scan of uint32 (any length up to 2^31): one block for up to
// SCAN_SMALL entries, three kernels beyond
// ---------------------------------------------------------------------------
constexpr int SCAN_T = 1024, SCAN_I = 4, SCAN_TILE = SCAN_T * SCAN_I;
// one block walks 4 tiles in about the time of the two further launches
constexpr int SCAN_SMALL = 4 * SCAN_TILE;

__device__ __forceinline__ unsigned block_excl_scan(unsigned v, unsigned *sw, unsigned *total)
{
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    unsigned x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        unsigned y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) sw[w] = x;
    __syncthreads();
    if (w == 0) {
        unsigned s = lane < nw ? sw[lane] : 0u;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            unsigned y = __shfl_up_sync(0xffffffffu, s, o);
            if (lane >= o) s += y;
        }
        if (lane < nw) sw[lane] = s;
    }
    __syncthreads();
    unsigned base = w ? sw[w - 1] : 0u;
    if (total) *total = sw[nw - 1];
    __syncthreads();
    return base + x - v;
}

__global__ void scan_reduce_k(const unsigned *__restrict__ in, int64_t n, unsigned *__restrict__ bsum)
{
    __shared__ unsigned sw[32];
    int64_t base = (int64_t)blockIdx.x * SCAN_TILE + (int64_t)threadIdx.x * SCAN_I;
    unsigned s = 0;
#pragma unroll
    for (int k = 0; k < SCAN_I; k++)
        if (base + k < n) s += in[base + k];
    unsigned tot;
    block_excl_scan(s, sw, &tot);
    if (threadIdx.x == 0) bsum[blockIdx.x] = tot;
}

__global__ void scan_top_k(unsigned *bsum, int nb, unsigned *total)
{
    __shared__ unsigned sw[32];
    unsigned carry = 0;
    for (int b0 = 0; b0 < nb; b0 += SCAN_T) {
        int i = b0 + threadIdx.x;
        unsigned v = i < nb ? bsum[i] : 0u;
        unsigned tot;
        unsigned ex = block_excl_scan(v, sw, &tot);
        if (i < nb) bsum[i] = carry + ex;
        carry += tot;
    }
    if (threadIdx.x == 0 && total) *total = carry;
}

__global__ void scan_apply_k(const unsigned *__restrict__ in, unsigned *__restrict__ out, int64_t n,
                             const unsigned *__restrict__ bsum)
{
    __shared__ unsigned sw[32];
    int64_t base = (int64_t)blockIdx.x * SCAN_TILE + (int64_t)threadIdx.x * SCAN_I;
    unsigned v[SCAN_I];
    unsigned s = 0;
#pragma unroll
    for (int k = 0; k < SCAN_I; k++) {
        v[k] = (base + k < n) ? in[base + k] : 0u;
        s += v[k];
    }
    unsigned ex = block_excl_scan(s, sw, nullptr) + bsum[blockIdx.x];
#pragma unroll
    for (int k = 0; k < SCAN_I; k++) {
        if (base + k < n) out[base + k] = ex;
        ex += v[k];
    }
}

__global__ void __launch_bounds__(SCAN_T) scan_small_k(const unsigned *__restrict__ in, unsigned *__restrict__ out, int n,
                                                       unsigned *total)
{
    __shared__ unsigned sw[32];
    unsigned carry = 0;
    for (int b0 = 0; b0 < n; b0 += SCAN_TILE) {
        const int base = b0 + (int)threadIdx.x * SCAN_I;
        unsigned v[SCAN_I], s = 0, tot;
#pragma unroll
        for (int k = 0; k < SCAN_I; k++) {
            v[k] = base + k < n ? in[base + k] : 0u;
            s += v[k];
        }
        unsigned ex = carry + block_excl_scan(s, sw, &tot);
#pragma unroll
        for (int k = 0; k < SCAN_I; k++) {
            if (base + k < n) out[base + k] = ex;
            ex += v[k];
        }
        carry += tot;
    }
    if (threadIdx.x == 0 && total) *total = carry;
}

void scan_exclusive_u32(fmm_ctx *h, const unsigned *in, unsigned *out, int64_t count, unsigned *total_dev,
                        cudaStream_t s)
{
    if (count <= 0) {
        if (total_dev) FMM_CUDA_TRY(cudaMemsetAsync(total_dev, 0, sizeof(unsigned), s));
        return;
    }
    if (count <= SCAN_SMALL) {
        scan_small_k<<<1, SCAN_T, 0, s>>>(in, out, (int)count, total_dev);
        count_launch(h);
        check_launch("scan");
        return;
    }
    int nb = (int)nblocks(count, SCAN_TILE);
    h->scan_tmp.ensure(sizeof(unsigned) * (size_t)(nb + 1));
    unsigned *bsum = h->scan_tmp.as<unsigned>();
    scan_reduce_k<<<nb, SCAN_T, 0, s>>>(in, count, bsum);
    count_launch(h);
    scan_top_k<<<1, SCAN_T, 0, s>>>(bsum, nb, total_dev);
    count_launch(h);
    scan_apply_k<<<nb, SCAN_T, 0, s>>>(in, out, count, bsum);
    count_launch(h);
    check_launch("scan");
}

// ---------------------------------------------------------------------------
// bounding cube and Morton keys
// ---------------------------------------------------------------------------
// FP32 -> FP64 without flushing subnormal inputs (the library is built with
// flush-to-zero for its FP32 arithmetic; the box and the keys use every
// input value exactly)
__device__ __forceinline__ double f32_to_f64_exact(float v)
{
    double d;
    asm("cvt.f64.f32 %0, %1;" : "=d"(d) : "f"(v));
    return d;
}
__device__ __forceinline__ double to_f64_exact(float v) { return f32_to_f64_exact(v); }
__device__ __forceinline__ double to_f64_exact(double v) { return v; }

// Extremes of the points i0, i0 + stride, ... < n over the whole block, as
// order-preserving encodings: e[0..2] the complements of the smallest, e[3..5]
// the largest coordinates (0: none seen), so that both are maxima and start at
// zero; bad: a coordinate was NaN or infinite. FP32 input stays in integer
// encodings of the float bits (exact, subnormals included, and off GB300's slow
// FP64 pipe) until one value per warp is left.
struct BoxAcc {
    unsigned long long e[32][6];
    int bad;
};
template <class T>
__device__ __forceinline__ void bbox_block(const T *__restrict__ x, int64_t n, int64_t i0, int64_t stride, BoxAcc &s,
                                           unsigned long long *enc)
{
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    int bad = 0;
    if (threadIdx.x == 0) s.bad = 0;
    unsigned long long e6[6] = {0, 0, 0, 0, 0, 0};
    if constexpr (sizeof(T) == 4) {
        // (no finite value encodes to 0xffffffff or to 0: the initial values mark "none seen")
        unsigned elo[3] = {0xffffffffu, 0xffffffffu, 0xffffffffu}, ehi[3] = {0u, 0u, 0u};
#pragma unroll 4
        for (int64_t i = i0; i < n; i += stride) {
#pragma unroll
            for (int k = 0; k < 3; k++) {
                const unsigned u = __float_as_uint((float)x[3 * i + k]);
                if ((u & 0x7f800000u) == 0x7f800000u) bad = 1;
                else {
                    const unsigned e = (u >> 31) ? ~u : (u | 0x80000000u);
                    elo[k] = min(elo[k], e);
                    ehi[k] = max(ehi[k], e);
                }
            }
        }
#pragma unroll
        for (int k = 0; k < 3; k++) {
            const unsigned lo = __reduce_min_sync(0xffffffffu, elo[k]), hi = __reduce_max_sync(0xffffffffu, ehi[k]);
            if (lane == 0 && lo != 0xffffffffu) {
                const unsigned a = (lo >> 31) ? (lo & 0x7fffffffu) : ~lo;
                const unsigned c = (hi >> 31) ? (hi & 0x7fffffffu) : ~hi;
                e6[k] = ~ord_enc(f32_to_f64_exact(__uint_as_float(a)));
                e6[3 + k] = ord_enc(f32_to_f64_exact(__uint_as_float(c)));
            }
        }
    } else {
        double lo[3] = {INFINITY, INFINITY, INFINITY}, hi[3] = {-INFINITY, -INFINITY, -INFINITY};
        for (int64_t i = i0; i < n; i += stride) {
#pragma unroll
            for (int k = 0; k < 3; k++) {
                const double v = (double)x[3 * i + k];
                if (!isfinite(v)) bad = 1;
                else {
                    lo[k] = fmin(lo[k], v);
                    hi[k] = fmax(hi[k], v);
                }
            }
        }
#pragma unroll
        for (int k = 0; k < 3; k++) {
            for (int o = 16; o > 0; o >>= 1) {
                lo[k] = fmin(lo[k], __shfl_xor_sync(0xffffffffu, lo[k], o));
                hi[k] = fmax(hi[k], __shfl_xor_sync(0xffffffffu, hi[k], o));
            }
            if (lo[k] <= hi[k]) {
                e6[k] = ~ord_enc(lo[k]);
                e6[3 + k] = ord_enc(hi[k]);
            }
        }
    }
    if (lane == 0)
        for (int k = 0; k < 6; k++) s.e[w][k] = e6[k];
    bad = __any_sync(0xffffffffu, bad);
    __syncthreads();
    if (bad && lane == 0) s.bad = 1;
    if (threadIdx.x < 6) {
        unsigned long long m = 0;
        for (int k = 0; k < nw; k++) m = max(m, s.e[k][threadIdx.x]);
        s.e[0][threadIdx.x] = m;
    }
    __syncthreads();
    for (int k = 0; k < 6; k++) enc[k] = s.e[0][k];
}

// Root cube from the bounding box, all in correctly rounded FP64:
// c = (lo + hi) / 2, R0 = max half extent (1 if 0), origin = c - R0,
// s = 2^21 / (2 R0), h = 2 R0 / 2^21.
__device__ __forceinline__ void box_finish(const unsigned long long *enc, Box *b)
{
    double R0 = 0.0, c[3];
    for (int k = 0; k < 6; k++) b->enc[k] = enc[k];
    for (int k = 0; k < 3; k++) {
        double lo = ord_dec(~enc[k]), hi = ord_dec(enc[3 + k]);
        c[k] = __dmul_rn(__dadd_rn(lo, hi), 0.5);
        double half = __dmul_rn(__dsub_rn(hi, lo), 0.5);
        if (half > R0) R0 = half;
    }
    if (R0 == 0.0) R0 = 1.0;
    for (int k = 0; k < 3; k++) b->origin[k] = __dsub_rn(c[k], R0);
    b->R0 = R0;
    b->s = __ddiv_rn(2097152.0, __dmul_rn(2.0, R0));
    b->h = __ddiv_rn(__dmul_rn(2.0, R0), 2097152.0);
}

// Bounding cube (b zeroed before): six atomics per block, and the last block to
// finish derives the cube. (Six atomics per warp took 46 us at n = 10^6.)
template <class T>
__global__ void __launch_bounds__(256) bbox_k(const T *__restrict__ x, int64_t n, Box *b)
{
    __shared__ BoxAcc s;
    __shared__ int last;
    unsigned long long enc[6];
    bbox_block(x, n, (int64_t)blockIdx.x * blockDim.x + threadIdx.x, (int64_t)gridDim.x * blockDim.x, s, enc);
    if (threadIdx.x < 6) {
        unsigned long long v = 0;
#pragma unroll
        for (int k = 0; k < 6; k++)
            if ((int)threadIdx.x == k) v = enc[k];
        if (v) atomicMax(&b->enc[threadIdx.x], v);
        if (threadIdx.x == 0 && s.bad) atomicOr(&b->nonfinite, 1);
        __threadfence();
    }
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(&b->ticket, 1u) == gridDim.x - 1;
    __syncthreads();
    if (last && threadIdx.x == 0) {
        __threadfence();
        for (int k = 0; k < 6; k++) enc[k] = __ldcg(&b->enc[k]);
        box_finish(enc, b);
    }
}

// i_k = clamp(floor((x_k - origin_k) * s), 0, 2^21 - 1); key interleaves
// x, y, z bits with x lowest.
template <class T>
__device__ __forceinline__ uint64_t morton_key(const T *__restrict__ x, int64_t i, const double (&org)[3], double s)
{
    uint32_t ic[3];
#pragma unroll
    for (int k = 0; k < 3; k++) {
        const double v = to_f64_exact(x[3 * i + k]);
        // floor to an integer in one conversion (saturating), clamped as an
        // integer: the same value as floor, clamp and cast in FP64, with half
        // the FP64 instructions
        const int f = __double2int_rd(__dmul_rn(__dsub_rn(v, org[k]), s));
        ic[k] = (uint32_t)min(max(f, 0), 2097151);
    }
    return morton3(ic[0], ic[1], ic[2]);
}

// ---------------------------------------------------------------------------
// stable LSD radix sort of 64-bit keys (8-bit digits) with int32 values
//
// The counts of all digits are taken in one read of the unsorted keys (for the
// Morton keys while they are made); a pass is then one kernel: a tile ranks
// its keys, publishes its digit counts and adds up those of the tiles before
// it ("decoupled look-back": Merrill and Garland, Single-pass parallel prefix
// scan with decoupled look-back, 2016; Adinets and Merrill, Onesweep, 2022).
// Bound: one read and one write of 12 bytes per key and pass. The passes as
// tile histograms, a scan of three kernels and a scatter took 376 us for
// n = 10^6 and 1.3 ms for 10^7; this takes 213 us and 1.1 ms.
// ---------------------------------------------------------------------------
constexpr int RS_T = 256, RS_W = RS_T / 32, RS_PASSES = 8;
constexpr int RS_R_MAX = 16;            // keys per thread: tiles of 4096 keys ...
constexpr int RS_R_MIN = 4;             // ... or of 1024 up to RS_FEW keys, so that every SM has one
constexpr int64_t RS_FEW = 1 << 19;
// workspace, all zero before a sort: digit counts, a tile counter per pass,
// then a status word per tile and digit
struct SortWs {
    unsigned count[RS_PASSES][256];
    unsigned ticket[RS_PASSES];
};
static int rs_tile(int64_t n) { return RS_T * (n <= RS_FEW ? RS_R_MIN : RS_R_MAX); }
// status: pass + 1 in the top 4 bits (a word left by another pass counts as not
// written), 1 (the tile's own count) or 2 (the count up to and including it) in
// the next two, the count in the rest: 26 bits, or 58 for more keys
static bool rs_wide(int64_t n) { return n >= (1 << 26); }
size_t sort_ws_bytes(int64_t n)
{
    return sizeof(SortWs) + (size_t)nblocks(n, rs_tile(n)) * 256 * (rs_wide(n) ? 8 : 4);
}

// Morton keys, with the counts of their 8 digits
template <class T>
__global__ void __launch_bounds__(256) keys_k(const T *__restrict__ x, int64_t n, const Box *__restrict__ b,
                                              uint64_t *__restrict__ keys, int *__restrict__ idx, SortWs *__restrict__ ws)
{
    __shared__ unsigned cnt[RS_PASSES * 256];
    for (int i = threadIdx.x; i < RS_PASSES * 256; i += 256) cnt[i] = 0;
    __syncthreads();
    const double org[3] = {b->origin[0], b->origin[1], b->origin[2]}, sc = b->s;
    for (int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x; i < n; i += (int64_t)gridDim.x * 256) {
        const uint64_t k = morton_key(x, i, org, sc);
        keys[i] = k;
        idx[i] = (int)i;
#pragma unroll
        for (int d = 0; d < RS_PASSES; d++) atomicAdd(&cnt[d * 256 + ((unsigned)(k >> (8 * d)) & 255u)], 1u);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < RS_PASSES * 256; i += 256)
        if (cnt[i]) atomicAdd(&ws->count[0][0] + i, cnt[i]);
}

// the digit counts of given keys
__global__ void __launch_bounds__(256) rs_count_k(const uint64_t *__restrict__ keys, int64_t n, int passes,
                                                  SortWs *__restrict__ ws)
{
    __shared__ unsigned cnt[RS_PASSES * 256];
    for (int i = threadIdx.x; i < RS_PASSES * 256; i += 256) cnt[i] = 0;
    __syncthreads();
    for (int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x; i < n; i += (int64_t)gridDim.x * 256) {
        const uint64_t k = keys[i];
        for (int d = 0; d < passes; d++) atomicAdd(&cnt[d * 256 + ((unsigned)(k >> (8 * d)) & 255u)], 1u);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < passes * 256; i += 256)
        if (cnt[i]) atomicAdd(&ws->count[0][0] + i, cnt[i]);
}

// the lanes whose 8-bit digit equals this lane's, by eight ballots (with match_any a
// sort of 10^6 keys takes 8 % longer)
__device__ __forceinline__ unsigned digit_peers(unsigned d)
{
    unsigned m = 0xffffffffu;
#pragma unroll
    for (int b = 0; b < 8; b++) {
        const unsigned v = __ballot_sync(0xffffffffu, (d >> b) & 1u);
        m &= ((d >> b) & 1u) ? v : ~v;
    }
    return m;
}

// how many of the first `base` keys have digit threadIdx.x (by the whole block; cnt:
// 256 words of its shared memory)
static __device__ __noinline__ unsigned rs_recount(const uint64_t *kin, int64_t base, int shift, unsigned *cnt)
{
    cnt[threadIdx.x] = 0;
    __syncthreads();
    for (int64_t i = threadIdx.x; i < base; i += RS_T) atomicAdd(&cnt[(unsigned)(kin[i] >> shift) & 255u], 1u);
    __syncthreads();
    return cnt[threadIdx.x];
}

// Each warp ranks its 32 R consecutive keys in R rounds of 32 (the lanes of
// equal digit by ballots), so the rank of a key among equal digits follows input order;
// the tile is staged in shared memory in digit order and written out in runs.
// Tiles are numbered in the order in which their blocks start, so a tile only
// waits for tiles that are already running. A tile that has looked more than `polls`
// times in vain for the one before counts the keys before its own itself: every wait
// is bounded, and the sort does not depend on one.
template <bool VALS, int R, class W>
__global__ void __launch_bounds__(RS_T) rs_pass_k(const uint64_t *__restrict__ kin, const int *__restrict__ vin,
                                                  uint64_t *__restrict__ kout, int *__restrict__ vout, int n, int pass,
                                                  SortWs *__restrict__ ws, W *status, int polls)
{
    constexpr int TILE = RS_T * R, CB = 8 * sizeof(W) - 6;  // bits of a count
    extern __shared__ unsigned char smem_raw[];
    uint64_t *skey = reinterpret_cast<uint64_t *>(smem_raw);               // TILE
    int *sval = reinterpret_cast<int *>(skey + TILE);                      // TILE
    unsigned *wcnt = reinterpret_cast<unsigned *>(sval + TILE);            // RS_W * 256
    unsigned *dstart = wcnt + RS_W * 256;                                  // 256
    unsigned *goff = dstart + 256;                                         // 256
    unsigned *sw = goff + 256;                                             // 32
    __shared__ unsigned s_tile;
    __shared__ int s_unknown;  // a thread gave up

    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, d0 = threadIdx.x, shift = 8 * pass;
    if (threadIdx.x == 0) {
        s_tile = atomicAdd(&ws->ticket[pass], 1u);
        s_unknown = 0;
    }
    for (int i = threadIdx.x; i < RS_W * 256; i += RS_T) wcnt[i] = 0;
    __syncthreads();
    const int tile = (int)s_tile;
    const int64_t base = (int64_t)tile * TILE;

    const unsigned lt = (1u << lane) - 1u;
    uint64_t k[R];
    int v[R];
    unsigned rank[R];
#pragma unroll
    for (int r = 0; r < R; r++) {
        const int64_t i = base + w * (32 * R) + r * 32 + lane;
        const bool ok = i < n;
        k[r] = ok ? kin[i] : ~0ull;
        v[r] = (VALS && ok) ? vin[i] : 0;
    }
#pragma unroll
    for (int r = 0; r < R; r++) {
        const unsigned d = (unsigned)(k[r] >> shift) & 255u;
        const unsigned peers = digit_peers(d);
        const unsigned c = wcnt[w * 256 + d];
        rank[r] = c + __popc(peers & lt);
        __syncwarp();
        if (lane == __ffs(peers) - 1) wcnt[w * 256 + d] = c + __popc(peers);
        __syncwarp();
    }
    __syncthreads();
    // per digit (thread d0): exclusive prefix over warps and the tile total
    unsigned run = 0;
#pragma unroll
    for (int ww = 0; ww < RS_W; ww++) {
        const unsigned c = wcnt[ww * 256 + d0];
        wcnt[ww * 256 + d0] = run;
        run += c;
    }
    // keys past n (the last tile's padding, all ones) are not counted
    const int64_t over = base + TILE - n;
    const unsigned own = run - (d0 == 255 && over > 0 ? (unsigned)over : 0u);
    const W tag = (W)(pass + 1) << (CB + 2);
    volatile W *st = status;
    st[(size_t)tile * 256 + d0] = tag | ((W)(tile == 0 ? 2 : 1) << CB) | (W)own;
    dstart[d0] = block_excl_scan(run, sw, nullptr);
    const unsigned gbase = block_excl_scan(ws->count[pass][d0], sw, nullptr);
    // the counts of the tiles before, eight words in flight
    unsigned before = 0;
    if (tile > 0) {
        constexpr int LB = 8;
        int t = tile - 1, n0 = 0;
        bool known = false;
        while (!known) {
            W x[LB];
#pragma unroll
            for (int j = 0; j < LB; j++) x[j] = t - j >= 0 ? st[(size_t)(t - j) * 256 + d0] : 0;
            bool go = true;
            int taken = 0;
#pragma unroll
            for (int j = 0; j < LB; j++) {
                go = go && (x[j] >> (CB + 2)) == (W)(pass + 1);
                if (go) {
                    before += (unsigned)(x[j] & (((W)1 << CB) - 1));
                    taken++;
                    known = ((x[j] >> CB) & 3) == 2;
                    go = !known;
                }
            }
            t -= taken;
            if (!known && taken == 0 && ++n0 > polls) break;
        }
        if (!known) s_unknown = 1;
        else st[(size_t)tile * 256 + d0] = tag | ((W)2 << CB) | (W)(before + own);
    }
    goff[d0] = gbase + before;
    __syncthreads();
    if (s_unknown) {
        before = rs_recount(kin, base, shift, reinterpret_cast<unsigned *>(skey));  // (not in use yet)
        st[(size_t)tile * 256 + d0] = tag | ((W)2 << CB) | (W)(before + own);
        goff[d0] = gbase + before;
        __syncthreads();
    }
#pragma unroll
    for (int r = 0; r < R; r++) {
        const unsigned d = (unsigned)(k[r] >> shift) & 255u;
        const unsigned pos = dstart[d] + wcnt[w * 256 + d] + rank[r];
        skey[pos] = k[r];
        if (VALS) sval[pos] = v[r];
    }
    __syncthreads();
    const int nvalid = (int)min((int64_t)TILE, n - base);
    for (int j = threadIdx.x; j < nvalid; j += RS_T) {
        const uint64_t kk = skey[j];
        const unsigned d = (unsigned)(kk >> shift) & 255u;
        const unsigned g = goff[d] + (unsigned)j - dstart[d];
        kout[g] = kk;
        if (VALS) vout[g] = sval[j];
    }
}

template <int R>
static size_t rs_smem() { return (size_t)RS_T * R * 12 + (size_t)(RS_W * 256 + 256 + 256 + 32) * 4; }

// Sorts by the low `bits` bits of the keys; ws holds their digit counts, zeros
// elsewhere. Returns true when the result sits in (kt, vt) rather than (k, v).
template <bool VALS, int R, class W>
static bool radix_passes(uint64_t *k, int *v, uint64_t *kt, int *vt, int n, int bits, SortWs *ws, int polls, cudaStream_t s)
{
    const int ntiles = (int)nblocks(n, RS_T * R);
    ensure_smem((const void *)rs_pass_k<VALS, R, W>, rs_smem<R>());
    bool swapped = false;
    for (int pass = 0; 8 * pass < bits; pass++) {
        rs_pass_k<VALS, R, W><<<ntiles, RS_T, rs_smem<R>(), s>>>(k, v, kt, vt, n, pass, ws, reinterpret_cast<W *>(ws + 1), polls);
        check_launch("radix sort");
        std::swap(k, kt);
        std::swap(v, vt);
        swapped = !swapped;
    }
    return swapped;
}

template <bool VALS>
static bool radix_sort(uint64_t *k, int *v, uint64_t *kt, int *vt, int64_t n, int bits, SortWs *ws, int polls, cudaStream_t s)
{
    if (n > 0x7fffffffLL) throw Error{FMM_EINVAL, "radix sort: too many keys"};
    if (rs_wide(n)) return radix_passes<VALS, RS_R_MAX, unsigned long long>(k, v, kt, vt, (int)n, bits, ws, polls, s);
    if (n <= RS_FEW) return radix_passes<VALS, RS_R_MIN, unsigned>(k, v, kt, vt, (int)n, bits, ws, polls, s);
    return radix_passes<VALS, RS_R_MAX, unsigned>(k, v, kt, vt, (int)n, bits, ws, polls, s);
}

// Up to SMALL_N points: cube, keys and all passes in one block (a launch per
// pass would cost more than the pass). Warp w holds keys 32 R w .. 32 R (w + 1)
// - 1 in R rounds, as in rs_pass_k.
constexpr int SMALL_T = 1024, SMALL_R = 4, SMALL_N = SMALL_T * SMALL_R;
constexpr size_t SMALL_SMEM = (size_t)SMALL_N * 12 + (SMALL_T / 32) * 256 * 2 + (256 + 32) * 4;
template <class T>
__global__ void __launch_bounds__(SMALL_T) sort_small_k(const T *__restrict__ x, int n, Box *__restrict__ b,
                                                        uint64_t *__restrict__ keys, int *__restrict__ perm)
{
    extern __shared__ unsigned char smem_raw[];
    uint64_t *skey = reinterpret_cast<uint64_t *>(smem_raw);
    int *sval = reinterpret_cast<int *>(skey + SMALL_N);
    unsigned *dstart = reinterpret_cast<unsigned *>(sval + SMALL_N);
    unsigned *sw = dstart + 256;
    unsigned short *wcnt = reinterpret_cast<unsigned short *>(sw + 32);  // [warp][256]
    __shared__ BoxAcc acc;
    __shared__ double s_org[4];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    {
        unsigned long long enc[6];
        bbox_block(x, (int64_t)n, (int64_t)threadIdx.x, (int64_t)SMALL_T, acc, enc);
        if (threadIdx.x == 0) {
            Box c;
            box_finish(enc, &c);
            c.nonfinite = acc.bad;
            c.ticket = 0;
            *b = c;
            for (int k = 0; k < 3; k++) s_org[k] = c.origin[k];
            s_org[3] = c.s;
        }
        __syncthreads();
    }
    const double org[3] = {s_org[0], s_org[1], s_org[2]}, sc = s_org[3];
    const int R = (n + SMALL_T - 1) / SMALL_T;
    const unsigned lt = (1u << lane) - 1u;
    uint64_t k[SMALL_R];
    int v[SMALL_R];
    unsigned rank[SMALL_R];
#pragma unroll
    for (int r = 0; r < SMALL_R; r++) {
        const int i = w * 32 * R + r * 32 + lane;
        k[r] = ~0ull;  // past n: after every key in each pass
        v[r] = i;
        if (r < R && i < n) k[r] = morton_key(x, i, org, sc);
    }
    for (int shift = 0; shift < 64; shift += 8) {
        for (int i = threadIdx.x; i < SMALL_T / 32 * 256; i += SMALL_T) wcnt[i] = 0;
        __syncthreads();
#pragma unroll
        for (int r = 0; r < SMALL_R; r++) {
            if (r >= R) break;
            const unsigned d = (unsigned)(k[r] >> shift) & 255u;
            const unsigned peers = digit_peers(d);
            const unsigned c = wcnt[w * 256 + d];
            rank[r] = c + __popc(peers & lt);
            __syncwarp();
            if (lane == __ffs(peers) - 1) wcnt[w * 256 + d] = (unsigned short)(c + __popc(peers));
            __syncwarp();
        }
        __syncthreads();
        unsigned run = 0;
        if (threadIdx.x < 256)
            for (int ww = 0; ww < SMALL_T / 32; ww++) {
                const unsigned c = wcnt[ww * 256 + threadIdx.x];
                wcnt[ww * 256 + threadIdx.x] = (unsigned short)run;
                run += c;
            }
        const unsigned ex = block_excl_scan(run, sw, nullptr);
        if (threadIdx.x < 256) dstart[threadIdx.x] = ex;
        __syncthreads();
#pragma unroll
        for (int r = 0; r < SMALL_R; r++) {
            if (r >= R) break;
            const unsigned d = (unsigned)(k[r] >> shift) & 255u;
            const unsigned pos = dstart[d] + wcnt[w * 256 + d] + rank[r];
            skey[pos] = k[r];
            sval[pos] = v[r];
        }
        __syncthreads();
#pragma unroll
        for (int r = 0; r < SMALL_R; r++) {
            if (r >= R) break;
            const int i = w * 32 * R + r * 32 + lane;
            k[r] = skey[i];
            v[r] = sval[i];
        }
        __syncthreads();
    }
#pragma unroll
    for (int r = 0; r < SMALL_R; r++) {
        const int i = w * 32 * R + r * 32 + lane;
        if (r < R && i < n) {
            keys[i] = k[r];
            perm[i] = v[r];
        }
    }
}

// Bounding cube, Morton keys and their stable sort into caller-provided
// buffers (no allocation; both the tree build and the allocation-free entry
// point): keys[n], perm[n] the sorted keys and the input index of each,
// keys_tmp, perm_tmp ping-pong buffers, ws sort_ws_bytes(n) of workspace. The
// result is in keys and perm (an even number of passes). polls: as in rs_pass_k.
// Returns the launches.
int morton_sort_into(const void *x, int64_t n, int dt, uint64_t *keys, int *perm, uint64_t *keys_tmp, int *perm_tmp,
                     void *ws, Box *box, int nsm, int polls, cudaStream_t s)
{
    const bool f64 = dt == FMM_F64;
    if (n <= SMALL_N) {
        ensure_smem(f64 ? (const void *)sort_small_k<double> : (const void *)sort_small_k<float>, SMALL_SMEM);
        if (f64) sort_small_k<double><<<1, SMALL_T, SMALL_SMEM, s>>>((const double *)x, (int)n, box, keys, perm);
        else sort_small_k<float><<<1, SMALL_T, SMALL_SMEM, s>>>((const float *)x, (int)n, box, keys, perm);
        check_launch("sort");
        return 1;
    }
    FMM_CUDA_TRY(cudaMemsetAsync(box, 0, sizeof(Box), s));
    FMM_CUDA_TRY(cudaMemsetAsync(ws, 0, sort_ws_bytes(n), s));
    SortWs *w = static_cast<SortWs *>(ws);
    // blocks: enough loads in flight for the box, 4096 keys or more per block
    // for the counts (2,048 atomics per block)
    const unsigned gb = (unsigned)std::min<int64_t>(nblocks(n, 1024), (int64_t)nsm * 8);
    const unsigned gk = (unsigned)std::min<int64_t>(nblocks(n, 2048), (int64_t)nsm * 6);
    if (f64) {
        bbox_k<double><<<gb, 256, 0, s>>>((const double *)x, n, box);
        keys_k<double><<<gk, 256, 0, s>>>((const double *)x, n, box, keys, perm, w);
    } else {
        bbox_k<float><<<gb, 256, 0, s>>>((const float *)x, n, box);
        keys_k<float><<<gk, 256, 0, s>>>((const float *)x, n, box, keys, perm, w);
    }
    check_launch("keys");
    radix_sort<true>(keys, perm, keys_tmp, perm_tmp, n, 63, w, polls, s);
    return 2 + RS_PASSES;
}

// Sorted particles (x, y, z, q). For the mixed path the FP32 copy holds the
// rounded coordinates, and xs32lo the FP32 rounding of the remainder x - hi
// (zero for FP32 inputs), so that a near-field difference can be formed as
// (hi_i - hi_j) + (lo_i - lo_j) without the rounding of the positions.
template <class T>
__global__ void gather_k(const T *__restrict__ x, const T *__restrict__ q, const int *__restrict__ idx, int64_t n,
                         double4_32a *__restrict__ xs64, float4 *__restrict__ xs32, float4 *__restrict__ xs32lo,
                         int *__restrict__ inv)
{
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    int j = idx[i];
    inv[j] = (int)i;
    const double a = to_f64_exact(x[3 * (int64_t)j]), b = to_f64_exact(x[3 * (int64_t)j + 1]),
                 c = to_f64_exact(x[3 * (int64_t)j + 2]);
    const double d = to_f64_exact(q[j]);
    if (xs64) xs64[i] = make_double4_32a(a, b, c, d);
    if (xs32) {
        const float ha = (float)a, hb = (float)b, hc = (float)c;
        xs32[i] = make_float4(ha, hb, hc, (float)d);
        if (xs32lo) xs32lo[i] = make_float4((float)(a - ha), (float)(b - hb), (float)(c - hc), 0.f);
    }
}

// ---------------------------------------------------------------------------
// cells: a cell of level l < 21 with more than ncrit particles splits into its
// non-empty octants, ascending octant order, numbered breadth first
// ---------------------------------------------------------------------------
__global__ void root_k(int n, int *level, uint64_t *anchor, int *begin, int *end, int *child, int *nchild,
                       int *parent, int4 *xyz)
{
    level[0] = 0;
    anchor[0] = 0;
    begin[0] = 0;
    end[0] = n;
    child[0] = -1;
    nchild[0] = 0;
    parent[0] = -1;
    xyz[0] = make_int4(0, 0, 0, 0);
}

// Eight lanes per cell, lane o searching the first key of octant o on its own:
// the searches of a cell are dependent loads of about 0.4 us each, so one
// thread doing the seven in turn takes 7 log2(range) of them (30 us a level for
// a handful of cells).
__global__ void split_count_k(int ls, int le, int l, int ncrit, const uint64_t *__restrict__ keys,
                              const int *__restrict__ begin, const int *__restrict__ end, unsigned *__restrict__ cnt,
                              int *__restrict__ bnd)
{
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    const int c = ls + (t >> 3), o = t & 7;
    const bool in = c < le;
    const int b = in ? begin[c] : 0, e = in ? end[c] : 0;
    const bool split = in && l < FMM_MAXLEVEL && e - b > ncrit;
    int L = b;
    if (split && o > 0) {
        const int shift = 3 * (FMM_MAXLEVEL - 1 - l);
        int H = e;  // first index with digit >= o
        while (L < H) {
            const int mid = L + ((H - L) >> 1);
            if ((int)((keys[mid] >> shift) & 7u) < o) L = mid + 1;
            else H = mid;
        }
    }
    int next = __shfl_down_sync(0xffffffffu, L, 1, 8);
    if (o == 7) next = e;
    const unsigned full = __ballot_sync(0xffffffffu, split && next > L);
    if (!in) return;
    if (split) {
        int *bb = bnd + (size_t)(c - ls) * 9;
        bb[o] = L;
        if (o == 7) bb[8] = e;
    }
    if (o == 0) cnt[c - ls] = __popc((full >> (threadIdx.x & 24)) & 0xffu);
}

__global__ void split_write_k(int ls, int le, int l, const unsigned *__restrict__ cnt, const unsigned *__restrict__ off,
                              const int *__restrict__ bnd, int *level, uint64_t *anchor, int *begin, int *end,
                              int *child, int *nchild, int *parent, int4 *xyz)
{
    int c = ls + blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= le) return;
    unsigned nc = cnt[c - ls];
    nchild[c] = (int)nc;
    child[c] = nc ? le + (int)off[c - ls] : -1;
    if (!nc) return;
    const int *bb = bnd + (size_t)(c - ls) * 9;
    const int shift = 3 * (FMM_MAXLEVEL - 1 - l);
    const int bit = FMM_MAXLEVEL - 1 - l;
    const int4 pxyz = xyz[c];
    const uint64_t pa = anchor[c];
    int k = le + (int)off[c - ls];
    for (int o = 0; o < 8; o++) {
        if (bb[o + 1] <= bb[o]) continue;
        level[k] = l + 1;
        anchor[k] = pa | ((uint64_t)o << shift);
        begin[k] = bb[o];
        end[k] = bb[o + 1];
        child[k] = -1;
        nchild[k] = 0;
        parent[k] = c;
        xyz[k] = make_int4(pxyz.x | ((o & 1) << bit), pxyz.y | (((o >> 1) & 1) << bit), pxyz.z | (((o >> 2) & 1) << bit),
                           l + 1);
        k++;
    }
}

// Small trees: every level's cells, the leaves, the leaf of each particle and
// the levels' lattice extents in one block. The general build takes three
// launches and a host round trip per level and seven launches after it; at N =
// 1,000 and 16,384 those were most of the build: 0.27 -> 0.16 ms and 0.50 ->
// 0.37 ms. Numbering and fields
// are those of the kernels above.
struct SmallTree {
    int nonfinite, overflow;
    int ncells, depth, nleaves;
    int lvl_start[FMM_MAXLEVEL + 2];
    int ext[6 * (FMM_MAXLEVEL + 1)];  // per level x y z: minima, then maxima
};
constexpr int TREE_SMALL_N = 32768;        // particles, and ...
constexpr int64_t TREE_SMALL_CELLS = 65536;  // ... cells that could arise (8 per cell over ncrit, 21 levels)
constexpr int TS_T = 1024;

__global__ void __launch_bounds__(TS_T) tree_small_k(int n, int ncrit, int cap, const uint64_t *__restrict__ keys,
                                                     const Box *__restrict__ box,
                                                     int *level, uint64_t *anchor, int *begin, int *end, int *child,
                                                     int *nchild, int *parent, int4 *xyz, int *leaves, int *pcell,
                                                     SmallTree *out)
{
    __shared__ unsigned s_cnt[TS_T / 8], s_off[TS_T / 8], sw[32];
    __shared__ int s_ext[6 * (FMM_MAXLEVEL + 1)];
    const int tid = threadIdx.x, o = tid & 7, lane = tid & 31;
    constexpr int NE = 3 * (FMM_MAXLEVEL + 1);
    for (int i = tid; i < 2 * NE; i += TS_T) s_ext[i] = i < NE ? INT_MAX : -1;
    if (tid == 0) {
        out->nonfinite = box->nonfinite;
        out->overflow = 0;
        level[0] = 0;
        anchor[0] = 0;
        begin[0] = 0;
        end[0] = n;
        parent[0] = -1;
        xyz[0] = make_int4(0, 0, 0, 0);
        out->lvl_start[0] = 0;
        out->lvl_start[1] = 1;
    }
    if (box->nonfinite) return;
    __syncthreads();
    int ls = 0, le = 1, l = 0;
    for (;; l++) {
        unsigned carry = 0;
        const int shift = 3 * (FMM_MAXLEVEL - 1 - l), bit = FMM_MAXLEVEL - 1 - l;
        for (int c0 = ls; c0 < le; c0 += TS_T / 8) {
            const int c = c0 + (tid >> 3);
            const bool in = c < le;
            const int b = in ? begin[c] : 0, e = in ? end[c] : 0;
            const bool split = in && l < FMM_MAXLEVEL && e - b > ncrit;
            int L = b;
            if (split && o > 0) {
                int H = e;  // first index with digit >= o
                while (L < H) {
                    const int mid = L + ((H - L) >> 1);
                    if ((int)((keys[mid] >> shift) & 7u) < o) L = mid + 1;
                    else H = mid;
                }
            }
            int next = __shfl_down_sync(0xffffffffu, L, 1, 8);
            if (o == 7) next = e;
            const bool some = split && next > L;
            const unsigned mine = (__ballot_sync(0xffffffffu, some) >> (lane & 24)) & 0xffu;
            const unsigned cnt = __popc(mine);
            if (o == 0) s_cnt[tid >> 3] = cnt;
            __syncthreads();
            unsigned tot;
            const unsigned ex = block_excl_scan(tid < TS_T / 8 ? s_cnt[tid] : 0u, sw, &tot);
            if (tid < TS_T / 8) s_off[tid] = ex;
            __syncthreads();
            const unsigned off = carry + s_off[tid >> 3];
            carry += tot;
            if ((int64_t)le + carry > cap) break;  // (the same in every thread)
            if (in && o == 0) {
                nchild[c] = (int)cnt;
                child[c] = cnt ? le + (int)off : -1;
            }
            if (some) {
                const int k = le + (int)off + __popc(mine & ((1u << o) - 1u));
                const int4 px = xyz[c];
                level[k] = l + 1;
                anchor[k] = anchor[c] | ((uint64_t)o << shift);
                begin[k] = L;
                end[k] = next;
                parent[k] = c;
                xyz[k] = make_int4(px.x | ((o & 1) << bit), px.y | (((o >> 1) & 1) << bit), px.z | (((o >> 2) & 1) << bit), l + 1);
            }
        }
        if ((int64_t)le + carry > cap) {
            if (tid == 0) out->overflow = 1;
            return;
        }
        __syncthreads();
        if (carry == 0) break;
        ls = le;
        le += (int)carry;
        if (tid == 0) out->lvl_start[l + 2] = le;
    }
    const int nc = le;
    unsigned nl = 0;
    for (int c0 = 0; c0 < nc; c0 += TS_T) {
        const int c = c0 + tid;
        const bool leaf = c < nc && nchild[c] == 0;
        unsigned tot;
        const unsigned ex = block_excl_scan(leaf ? 1u : 0u, sw, &tot);
        if (leaf) leaves[nl + ex] = c;
        nl += tot;
        if (c < nc) {
            const int4 a = xyz[c];
            const int sh = FMM_MAXLEVEL - a.w;
            const int v[3] = {a.x >> sh, a.y >> sh, a.z >> sh};
            for (int k = 0; k < 3; k++) {
                atomicMin(&s_ext[3 * a.w + k], v[k]);
                atomicMax(&s_ext[NE + 3 * a.w + k], v[k]);
            }
        }
    }
    for (int c = tid >> 5; c < nc; c += TS_T / 32)
        if (nchild[c] == 0)
            for (int j = begin[c] + lane; j < end[c]; j += 32) pcell[j] = c;
    __syncthreads();
    for (int i = tid; i < 2 * NE; i += TS_T) out->ext[i] = s_ext[i];
    if (tid == 0) {
        out->ncells = nc;
        out->depth = l;
        out->nleaves = (int)nl;
    }
}

// ---------------------------------------------------------------------------
// dual traversal, one level of the pair frontier per launch
// ---------------------------------------------------------------------------

// Multipole acceptance in integer half-grid units: the box of level l is
// W = 2^(21-l) grid units wide, its centre 2*anchor + W half units, its half
// diagonal sqrt(3) W. Accept iff 3 (W_A + W_B)^2 < fl(theta^2 d^2).
__device__ __forceinline__ bool mac_accept(int4 a, int4 b, double c)
{
    const long long WA = 1LL << (FMM_MAXLEVEL - a.w), WB = 1LL << (FMM_MAXLEVEL - b.w);
    const long long dx = 2LL * (a.x - b.x) + (WA - WB);
    const long long dy = 2LL * (a.y - b.y) + (WA - WB);
    const long long dz = 2LL * (a.z - b.z) + (WA - WB);
    const long long d2 = dx * dx + dy * dy + dz * dz;
    const double lhs = __dmul_rn(3.0, (double)((WA + WB) * (WA + WB)));
    const double rhs = __dmul_rn(c, (double)d2);
    return lhs < rhs;
}

// The same test for two cells of one level: with W_A = W_B = W both sides
// carry the exact factor 4 W^2, so it reduces to 3 < fl(theta^2 |v|^2), v the
// offset in cell units, and by monotone rounding to |v|^2 >= K0 with K0 the
// first integer that passes (computed on the host with the same FP64 multiply).
__device__ __forceinline__ bool mac_accept_same(int4 a, int4 b, long long K0)
{
    const int sh = FMM_MAXLEVEL - a.w;
    const long long vx = (b.x - a.x) >> sh, vy = (b.y - a.y) >> sh, vz = (b.z - a.z) >> sh;
    return vx * vx + vy * vy + vz * vz >= K0;
}

// Per level, the smallest and largest lattice coordinate of the existing
// cells (ext[0..66): minima, level-major x y z; ext[66..132): maxima). Lanes
// of one level reduce in the warp first; cells are level-contiguous.
__global__ void extent_k(int nc, const int4 *__restrict__ xyz, int *__restrict__ ext)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const bool in = i < nc;
    const int4 a = in ? xyz[i] : make_int4(0, 0, 0, 0);
    const int l = in ? a.w : -1;
    const unsigned grp = __match_any_sync(0xffffffffu, l);
    if (!in) return;
    const int sh = FMM_MAXLEVEL - l;
    const int x = a.x >> sh, y = a.y >> sh, z = a.z >> sh;
    const int mnx = __reduce_min_sync(grp, x), mny = __reduce_min_sync(grp, y), mnz = __reduce_min_sync(grp, z);
    const int mxx = __reduce_max_sync(grp, x), mxy = __reduce_max_sync(grp, y), mxz = __reduce_max_sync(grp, z);
    if ((int)(threadIdx.x & 31) == __ffs(grp) - 1) {
        int *mn = ext + 3 * l, *mx = ext + 3 * (FMM_MAXLEVEL + 1) + 3 * l;
        atomicMin(mn, mnx);
        atomicMin(mn + 1, mny);
        atomicMin(mn + 2, mnz);
        atomicMax(mx, mxx);
        atomicMax(mx + 1, mxy);
        atomicMax(mx + 2, mxz);
    }
}

// One thread per (frontier pair, slot): the pair (A, B) expands into at most
// 8 x 8 child pairs; slot k takes child a = child[A] + k of A (or A itself)
// against the children of B (or B itself), at most 8 pairs, classified in
// registers and written after one reservation of the block per list. The
// atomics on the four counters bound it: with one per warp and list the build at
// N = 1e6 Plummer took 2.54 ms, with one per block 2.11 ms.
constexpr int EXPAND_T = 256;
__global__ void __launch_bounds__(EXPAND_T) expand_k(const int2 *__restrict__ F, unsigned nF, const int4 *__restrict__ xyz,
                                                const int *__restrict__ child, const int *__restrict__ nchild, double cm,
                                                long long K0,
                                                int2 *__restrict__ p2p, unsigned long long cap_p2p,
                                                int2 *__restrict__ m2lx, unsigned long long cap_m2lx,
                                                int2 *__restrict__ next, unsigned long long cap_next,
                                                TravCounters *ctr)
{
    const unsigned long long t = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x;
    const unsigned i = (unsigned)(t >> 3), slot = (unsigned)(t & 7);
    int a = -1, b0 = 0, nb = 0;
    if (i < nF) {
        const int2 pr = F[i];
        const int A = pr.x, B = pr.y;
        const int ncA = nchild[A], ncB = nchild[B];
        const int lA = xyz[A].w, lB = xyz[B].w;
        const bool la = ncA == 0, lb = ncB == 0;
        if (!la && (lb || lA < lB)) {  // split A only
            if ((int)slot < ncA) { a = child[A] + slot; b0 = B; nb = 1; }
        } else if (!lb && (la || lB < lA)) {  // split B only
            if (slot == 0) { a = A; b0 = child[B]; nb = ncB; }
        } else {  // both, same level
            if ((int)slot < ncA) { a = child[A] + slot; b0 = child[B]; nb = ncB; }
        }
    }
    unsigned mP = 0, mX = 0, mN = 0, cI = 0;
    if (a >= 0) {
        const int4 xa = xyz[a];
        const bool leafa = nchild[a] == 0;
        for (int k = 0; k < nb; k++) {
            const int b = b0 + k;
            const int4 xb = xyz[b];
            if (xa.w == xb.w ? mac_accept_same(xa, xb, K0) : mac_accept(xa, xb, cm)) {
                if (xa.w == xb.w) cI++;
                else mX |= 1u << k;
            } else if (leafa && nchild[b] == 0) mP |= 1u << k;
            else mN |= 1u << k;
        }
    }
    // the four counts as 16-bit fields (at most 8 a thread, 2,048 a block), in
    // the order of the counters
    constexpr int NW = EXPAND_T / 32;
    __shared__ unsigned long long wsum[NW], base[4];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned long long cnt = (unsigned long long)((unsigned)__popc(mP) | (unsigned)__popc(mX) << 16) |
                                   (unsigned long long)((unsigned)__popc(mN) | cI << 16) << 32;
    unsigned long long sum = cnt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long y = __shfl_up_sync(0xffffffffu, sum, o);
        if (lane >= o) sum += y;
    }
    if (lane == 31) wsum[warp] = sum;
    __syncthreads();
    unsigned long long before = 0, all = 0;
#pragma unroll
    for (int w = 0; w < NW; w++) {
        if (w == warp) before = all;
        all += wsum[w];
    }
    if (threadIdx.x < 4) {
        const unsigned long long c = (all >> (16 * threadIdx.x)) & 0xffffull;
        base[threadIdx.x] = c ? atomicAdd(reinterpret_cast<unsigned long long *>(ctr) + threadIdx.x, c) : 0ull;
    }
    __syncthreads();
    before += sum - cnt;
    unsigned long long oP = base[0] + (before & 0xffffull), oX = base[1] + ((before >> 16) & 0xffffull),
                       oN = base[2] + ((before >> 32) & 0xffffull);
    for (; mP; mP &= mP - 1, oP++)
        if (oP < cap_p2p) p2p[oP] = make_int2(a, b0 + __ffs(mP) - 1);
    for (; mX; mX &= mX - 1, oX++)
        if (oX < cap_m2lx) m2lx[oX] = make_int2(a, b0 + __ffs(mX) - 1);
    for (; mN; mN &= mN - 1, oN++)
        if (oN < cap_next) next[oN] = make_int2(a, b0 + __ffs(mN) - 1);
}

// ---------------------------------------------------------------------------
// pair lists -> CSR (sorted by target, then source)
// ---------------------------------------------------------------------------
__global__ void pair_keys_k(const int2 *__restrict__ pr, int64_t np, int bs, uint64_t *__restrict__ keys)
{
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= np) return;
    int2 v = pr[i];
    keys[i] = ((uint64_t)(unsigned)v.x << bs) | (uint64_t)(unsigned)v.y;
}

__global__ void pair_rows_k(const uint64_t *__restrict__ keys, int64_t np, int bs, unsigned *__restrict__ rowcnt,
                            int *__restrict__ src)
{
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= np) return;
    uint64_t k = keys[i];
    src[i] = (int)(k & ((1ull << bs) - 1));
    const int row = (int)(k >> bs);
    const unsigned same = __match_any_sync(__activemask(), row);
    if ((int)(threadIdx.x & 31) == __ffs(same) - 1) atomicAdd(&rowcnt[row], (unsigned)__popc(same));
}

// P2P source leaves of a target leaf that are adjacent in the sorted particle
// order are merged into runs [begin, end); runs of leaf A are stored at
// [ptr[A], ptr[A] + nrun[A]) of the run array (never more runs than leaves).
// With pad and flag (packed P2P) the runs are in records: particles [b, e) are
// records [(b + pad[b]) / 2, (e + pad[e - 1] + flag[e - 1]) / 2). One warp per
// leaf: an entry opens a run when it does not begin where its predecessor
// ends, and closes it when its successor does not begin where it ends; ballots
// number the runs. (One thread per leaf, its loads in turn, took 0.38 ms for
// 4,096 leaves of 250 sources and 0.74 ms for 53,000 of 178.) The entries'
// particle counts add up to the number of interactions.
constexpr int RUN_WARPS = 8;
__global__ void __launch_bounds__(32 * RUN_WARPS) p2p_runs_k(int nleaves, const int *__restrict__ leaves,
                                                             const int *__restrict__ ptr, const int *__restrict__ src,
                                                             const int *__restrict__ begin, const int *__restrict__ end,
                                                             const unsigned *__restrict__ pad,
                                                             const unsigned *__restrict__ flag, int2 *__restrict__ runs,
                                                             int *__restrict__ nrun, unsigned long long *inter)
{
    __shared__ unsigned long long ssum[RUN_WARPS];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int i = blockIdx.x * RUN_WARPS + w;
    unsigned long long sum = 0;
    if (i < nleaves) {
        const int A = leaves[i], k0 = ptr[A], k1 = ptr[A + 1];
        int o = k0;
        for (int kb = k0; kb < k1; kb += 32) {
            const int k = kb + lane;
            bool open = false, close = false;
            int b = 0, e = 0;
            if (k < k1) {
                const int s = src[k];
                b = begin[s];
                e = end[s];
                open = k == k0 || end[src[k - 1]] != b;
                close = k + 1 == k1 || begin[src[k + 1]] != e;
                sum += (unsigned long long)(e - b);
            }
            const unsigned m = __ballot_sync(0xffffffffu, open);
            const int pos = o + __popc(m & (0xffffffffu >> (31 - lane))) - 1;  // run of this entry
            if (open) runs[pos].x = pad ? (int)((b + pad[b]) >> 1) : b;
            if (close) runs[pos].y = pad ? (int)((e + pad[e - 1] + flag[e - 1]) >> 1) : e;
            o += __popc(m);
        }
        if (lane == 0) nrun[A] = o - k0;
        for (int d = 16; d > 0; d >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, d);
        sum *= (unsigned long long)(end[A] - begin[A]);
    }
    if (lane == 0) ssum[w] = sum;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int k = 1; k < RUN_WARPS; k++) sum += ssum[k];
        if (sum) atomicAdd(inter, sum);
    }
}

// (target, source) pairs -> CSR rows without a global sort: rows are counted
// and filled with warp-aggregated atomics, then each row is put in ascending
// source order by exact ranks (sources of a row are distinct).
__global__ void row_count_k(const int2 *__restrict__ pr, int64_t np, unsigned *__restrict__ cnt)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= np) return;
    const int a = pr[i].x;
    const unsigned act = __activemask();
    const unsigned same = __match_any_sync(act, a);
    if ((int)(threadIdx.x & 31) == __ffs(same) - 1) atomicAdd(&cnt[a], (unsigned)__popc(same));
}

__global__ void row_fill_k(const int2 *__restrict__ pr, int64_t np, const int *__restrict__ ptr, unsigned *__restrict__ cur,
                           int *__restrict__ src)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= np) return;
    const int2 v = pr[i];
    const unsigned act = __activemask();
    const unsigned same = __match_any_sync(act, v.x);
    const int lane = threadIdx.x & 31, leader = __ffs(same) - 1;
    unsigned base = 0;
    if (lane == leader) base = atomicAdd(&cur[v.x], (unsigned)__popc(same));
    base = __shfl_sync(same, base, leader);
    const unsigned rank = __popc(same & ((1u << lane) - 1));
    src[ptr[v.x] + base + rank] = v.y;
}

__global__ void row_max_k(int nc, const unsigned *__restrict__ cnt, unsigned *__restrict__ mx)
{
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    unsigned v = c < nc ? cnt[c] : 0u;
    for (int o = 16; o > 0; o >>= 1) v = max(v, __shfl_xor_sync(0xffffffffu, v, o));
    if ((threadIdx.x & 31) == 0 && v) atomicMax(mx, v);
}

constexpr int ROW_SORT_WARPS = 8, ROW_SORT_CAP = 1024;

// Ascending bitonic sort of 32 R keys held by one warp, lane l holding keys
// R l .. R l + R - 1: partners R or more apart are exchanged with shuffles, the
// others inside the lane's registers.
template <int R>
__device__ __forceinline__ void warp_bitonic(int (&v)[R], int lane)
{
#pragma unroll
    for (int k = 2; k <= 32 * R; k <<= 1) {
#pragma unroll
        for (int j = k >> 1; j > 0; j >>= 1) {
            if (j >= R) {
#pragma unroll
                for (int r = 0; r < R; r++) {
                    const int i = lane * R + r;
                    const int y = __shfl_xor_sync(0xffffffffu, v[r], j / R);
                    const bool up = (i & k) == 0, low = (i & j) == 0;
                    v[r] = low == up ? min(v[r], y) : max(v[r], y);
                }
            } else {
#pragma unroll
                for (int r = 0; r < R; r++) {
                    if (r & j) continue;
                    const bool up = ((lane * R + r) & k) == 0;
                    const int a = v[r], b = v[r | j];
                    v[r] = up ? min(a, b) : max(a, b);
                    v[r | j] = up ? max(a, b) : min(a, b);
                }
            }
        }
    }
}

template <int R>
__device__ __forceinline__ void row_sort_warp(int *src, int len, int lane)
{
    int v[R];
#pragma unroll
    for (int k = 0; k < R; k++) v[k] = lane * R + k < len ? src[lane * R + k] : INT_MAX;
    warp_bitonic<R>(v, lane);
#pragma unroll
    for (int k = 0; k < R; k++)
        if (lane * R + k < len) src[lane * R + k] = v[k];
}

// Each CSR row of up to ROW_SORT_CAP entries in ascending order, one warp per
// row, by a bitonic sort in registers of the next of 256, 512 and 1024 entries.
__global__ void __launch_bounds__(32 * ROW_SORT_WARPS) row_sort_k(int nc, const int *__restrict__ ptr, int *__restrict__ src)
{
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int r = blockIdx.x * ROW_SORT_WARPS + w;
    if (r >= nc) return;
    const int b = ptr[r], len = ptr[r + 1] - b;
    if (len <= 1 || len > ROW_SORT_CAP) return;
    if (len <= 256) row_sort_warp<8>(src + b, len, lane);
    else if (len <= 512) row_sort_warp<16>(src + b, len, lane);
    else row_sort_warp<32>(src + b, len, lane);
}

// ---------------------------------------------------------------------------
// uniform-tree fast path: on a full octree (every leaf on level L, every level
// full) the traversal's P2P lists are the near-field lattice stencil of level
// L, cut at the lattice boundary; cell id = first cell of level L + Morton
// index of the lattice position.  The traversal reaches a pair of leaves only
// if every pair of their ancestors was rejected; that holds for every near
// pair: theta < 1 gives K0 >= 4, and a child offset with |v|^2 <= K0 - 1 has a
// parent offset with |u_d| <= (|v_d| + 1) / 2, so
// |u|^2 <= (|v|^2 + 2 sqrt(3) |v| + 3) / 4 < K0.
// ---------------------------------------------------------------------------
// One warp per cell, its lanes over the stencil. Row counts into cnt[c] ...
__global__ void __launch_bounds__(256) near_count_k(int ls, int le, int L, const int4 *__restrict__ xyz,
                                                    const int4 *__restrict__ near, int nnear, unsigned *__restrict__ cnt)
{
    const int lane = threadIdx.x & 31, c = ls + (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5);
    if (c >= le) return;
    const int sh = FMM_MAXLEVEL - L;
    const unsigned side = 1u << L;
    const int4 a = xyz[c];
    const int px = a.x >> sh, py = a.y >> sh, pz = a.z >> sh;
    int k = 0;
    for (int e = lane; e < nnear; e += 32) {
        const int4 v = near[e];
        k += (unsigned)(px + v.x) < side && (unsigned)(py + v.y) < side && (unsigned)(pz + v.z) < side;
    }
    k = __reduce_add_sync(0xffffffffu, k);
    if (lane == 0) cnt[c] = (unsigned)k;
}

// ... and the rows at ptr[c], sorted in registers before they are written
// (32 R >= nnear; positions outside the lattice sort to the end)
template <int R>
__global__ void __launch_bounds__(256) near_rows_k(int ls, int le, int L, const int4 *__restrict__ xyz,
                                                   const int4 *__restrict__ near, int nnear, const int *__restrict__ ptr,
                                                   int *__restrict__ src)
{
    const int lane = threadIdx.x & 31, c = ls + (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5);
    if (c >= le) return;
    const int sh = FMM_MAXLEVEL - L;
    const unsigned side = 1u << L;
    const int4 a = xyz[c];
    const int px = a.x >> sh, py = a.y >> sh, pz = a.z >> sh;
    int v[R];
#pragma unroll
    for (int r = 0; r < R; r++) {
        const int e = 32 * r + lane;
        v[r] = INT_MAX;
        if (e < nnear) {
            const int4 d = near[e];
            const unsigned qx = (unsigned)(px + d.x), qy = (unsigned)(py + d.y), qz = (unsigned)(pz + d.z);
            if (qx < side && qy < side && qz < side) v[r] = ls + (int)morton3(qx, qy, qz);
        }
    }
    warp_bitonic<R>(v, lane);
    const int b = ptr[c], len = ptr[c + 1] - b;
#pragma unroll
    for (int r = 0; r < R; r++)
        if (lane * R + r < len) src[b + lane * R + r] = v[r];
}

static int bits_for(int64_t v)
{
    int b = 1;
    while ((1LL << b) <= v) b++;
    return b;
}

// Sort np (target, source) pairs into CSR rows over ncells cells.
static void pairs_to_csr(fmm_ctx *h, const int2 *pairs, int64_t np, DevBuf &ptr, DevBuf &src, cudaStream_t s)
{
    const int nc = h->ncells;
    ptr.ensure(sizeof(int) * (size_t)(nc + 1));
    src.ensure(sizeof(int) * (size_t)std::max<int64_t>(np, 1));
    h->row_cnt.ensure(sizeof(unsigned) * (size_t)(nc + 1));
    FMM_CUDA_TRY(cudaMemsetAsync(h->row_cnt.p, 0, sizeof(unsigned) * (size_t)(nc + 1), s));
    if (np > 0) {
        row_count_k<<<nblocks(np, 256), 256, 0, s>>>(pairs, np, h->row_cnt.as<unsigned>());
        count_launch(h);
        // longest row: rows that fit the per-warp sort are filled and ranked
        // in place, otherwise the pairs go through a global sort
        unsigned *dmax = reinterpret_cast<unsigned *>(h->counters.as<char>() + sizeof(TravCounters) + 32);
        FMM_CUDA_TRY(cudaMemsetAsync(dmax, 0, sizeof(unsigned), s));
        row_max_k<<<nblocks(nc, 256), 256, 0, s>>>(nc, h->row_cnt.as<unsigned>(), dmax);
        count_launch(h);
        unsigned *hp = h->hpin.as<unsigned>();
        FMM_CUDA_TRY(cudaMemcpyAsync(hp, dmax, sizeof(unsigned), cudaMemcpyDeviceToHost, s));
        FMM_CUDA_TRY(cudaStreamSynchronize(s));
        if (*hp <= (unsigned)ROW_SORT_CAP) {
            scan_exclusive_u32(h, h->row_cnt.as<unsigned>(), reinterpret_cast<unsigned *>(ptr.as<int>()), nc + 1, nullptr, s);
            FMM_CUDA_TRY(cudaMemsetAsync(h->row_cnt.p, 0, sizeof(unsigned) * (size_t)(nc + 1), s));
            row_fill_k<<<nblocks(np, 256), 256, 0, s>>>(pairs, np, ptr.as<int>(), h->row_cnt.as<unsigned>(), src.as<int>());
            count_launch(h);
            row_sort_k<<<nblocks(nc, ROW_SORT_WARPS), 32 * ROW_SORT_WARPS, 0, s>>>(nc, ptr.as<int>(), src.as<int>());
            count_launch(h);
            check_launch("pairs to csr");
            return;
        }
        FMM_CUDA_TRY(cudaMemsetAsync(h->row_cnt.p, 0, sizeof(unsigned) * (size_t)(nc + 1), s));
        const int bs = bits_for(nc - 1);
        h->pair_keys.ensure(sizeof(uint64_t) * (size_t)np);
        h->pair_keys2.ensure(sizeof(uint64_t) * (size_t)np);
        uint64_t *k1 = h->pair_keys.as<uint64_t>(), *k2 = h->pair_keys2.as<uint64_t>();
        pair_keys_k<<<nblocks(np, 256), 256, 0, s>>>(pairs, np, bs, k1);
        count_launch(h);
        h->sort_ws.ensure(sort_ws_bytes(np));
        SortWs *ws = h->sort_ws.as<SortWs>();
        FMM_CUDA_TRY(cudaMemsetAsync(ws, 0, sort_ws_bytes(np), s));
        rs_count_k<<<std::min(nblocks(np, 2048), (unsigned)h->nsm * 6), 256, 0, s>>>(k1, np, (2 * bs + 7) / 8, ws);
        count_launch(h);
        const bool sw = radix_sort<false>(k1, nullptr, k2, nullptr, np, 2 * bs, ws, h->sort_polls, s);
        h->launches += (2 * bs + 7) / 8;
        const uint64_t *ks = sw ? k2 : k1;
        pair_rows_k<<<nblocks(np, 256), 256, 0, s>>>(ks, np, bs, h->row_cnt.as<unsigned>(), src.as<int>());
        count_launch(h);
        check_launch("pairs to csr");
    }
    scan_exclusive_u32(h, h->row_cnt.as<unsigned>(), reinterpret_cast<unsigned *>(ptr.as<int>()), nc + 1, nullptr, s);
}

// ---------------------------------------------------------------------------
// per-level lattice maps and M2L target tiles
// ---------------------------------------------------------------------------
__global__ void map_fill_k(int ls, int le, int l, const uint64_t *__restrict__ anchor, int *__restrict__ map)
{
    int c = ls + blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= le) return;
    map[anchor[c] >> (3 * (FMM_MAXLEVEL - l))] = c;
}

// the cells of a level into the bricks of their ancestors `up` levels above,
// whose dense map is `top`
__global__ void brick_fill_k(int ls, int le, int l, int up, int top_start, const uint64_t *__restrict__ anchor,
                             const int *__restrict__ top, int *__restrict__ bricks)
{
    int c = ls + blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= le) return;
    const uint64_t k = anchor[c] >> (3 * (FMM_MAXLEVEL - l));
    const int a = top[k >> (3 * up)];
    bricks[((long long)(a - top_start) << (3 * up)) + (long long)(k & ((1ull << (3 * up)) - 1ull))] = c;
}

// the cells of a level without a map into its open-addressed table
// (linear probing; at most half full, so every insertion finds a slot)
__global__ void hash_fill_k(int ls, int le, int l, const uint64_t *__restrict__ anchor, HashSlot *__restrict__ tab,
                            unsigned mask)
{
    int c = ls + blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= le) return;
    const unsigned long long key = (anchor[c] >> (3 * (FMM_MAXLEVEL - l))) + 1ull;
    unsigned hs = level_hash(key, mask);
    for (unsigned i = 0; i <= mask; i++, hs = (hs + 1) & mask) {
        const unsigned long long prev = atomicCAS(&tab[hs].key, 0ull, key);
        if (prev == 0ull || prev == key) {
            tab[hs].val = c;
            return;
        }
    }
}

__global__ void oct_count_k(int c0, int nc, const int *__restrict__ level, const uint64_t *__restrict__ anchor,
                            unsigned *__restrict__ grp)
{
    int c = c0 + blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= nc) return;
    int l = level[c];
    int o = (int)((anchor[c] >> (3 * (FMM_MAXLEVEL - l))) & 7u);
    atomicAdd(&grp[l * 8 + o], 1u);
}

// One thread: group offsets and tile descriptors, levels 2..depth.
// Levels with at most pool_max cells would leave the tiles of their octant
// groups mostly empty: their cells (every octant) are pooled, level by level,
// at the front of the target list and cut into tiles of octant 8, whose
// level is the largest level among their cells. Within a denser level the
// tiles of the 8 octant groups are interleaved (tile k of octant 0, tile k of
// octant 1, ...), so that tiles running at the same time cover one compact
// region and share sources in L2.
// Lattice levels (bit l of lat) take every position of the level, cells or not,
// so that each tile is one block of its octant's sub-lattice.
__global__ void tiles_k(int depth, int tile, int pool_max, unsigned lat, const unsigned *__restrict__ grp,
                        unsigned *__restrict__ goff, M2LTile *__restrict__ tiles, int *__restrict__ ntiles)
{
    unsigned run = 0;
    int nt = 0;
    auto level_cells = [&](int l) {
        unsigned c = 0;
        for (int o = 0; o < 8; o++) c += grp[l * 8 + o];
        return c;
    };
    for (int l = 2; l <= depth; l++) {
        if (level_cells(l) > (unsigned)pool_max) continue;
        for (int o = 0; o < 8; o++) {
            goff[l * 8 + o] = run;
            run += grp[l * 8 + o];
        }
    }
    const unsigned pool = run;
    int lv = 2;
    for (unsigned t = 0; t < pool; t += tile) {
        const unsigned cnt = min((unsigned)tile, pool - t), last = t + cnt - 1;
        // level of the tile's last cell: the pooled levels are in ascending order
        while (lv < depth) {
            const unsigned c = level_cells(lv);
            if (c <= (unsigned)pool_max && c > 0 && last < goff[lv * 8] + c) break;
            lv++;
        }
        M2LTile d;
        d.start = (int)t;
        d.count = (int)cnt;
        d.level = lv;
        d.octant = 8;
        d.block = -1;
        tiles[nt++] = d;
    }
    for (int l = 2; l <= depth; l++) {
        if (level_cells(l) <= (unsigned)pool_max) continue;
        unsigned kmax = 0;
        for (int o = 0; o < 8; o++) {
            const unsigned c = (lat >> l) & 1u ? 1u << (3 * (l - 1)) : grp[l * 8 + o];
            goff[l * 8 + o] = run;
            run += c;
            kmax = max(kmax, (c + tile - 1) / tile);
        }
        for (unsigned k = 0; k < kmax; k++)
            for (int o = 0; o < 8; o++) {
                const unsigned c = (lat >> l) & 1u ? 1u << (3 * (l - 1)) : grp[l * 8 + o], t = k * tile;
                if (t >= c) continue;
                M2LTile d;
                d.start = (int)(goff[l * 8 + o] + t);
                d.count = (int)min((unsigned)tile, c - t);
                d.level = l;
                d.octant = o;
                d.block = (lat >> l) & 1u ? (int)k : -1;
                tiles[nt++] = d;
            }
    }
    *ntiles = nt;
}

// A complete (level, octant) group (all 8^(l-1) cells present) is placed in
// the Morton order of its sub-lattice, so that every 128 consecutive entries
// are a block of 8 x 4 x 4 cells (x taking Morton bits 0, 3, 6, y 1, 4 and z
// 2, 5 of the halved position). With raster set (tiles of 128 rows) the
// entries inside each such block of a group of at least 512 cells are put in
// x, y, z order, row = x + 8 y + 32 z, the order in which the tensor-core M2L
// loads a shifted block of sources by TMA. Other groups in arrival order.
__global__ void oct_scatter_k(int c0, int nc, const int *__restrict__ level, const uint64_t *__restrict__ anchor,
                              const unsigned *__restrict__ grp, const unsigned *__restrict__ goff,
                              unsigned *__restrict__ fill, int raster, unsigned lat, int *__restrict__ tgt)
{
    int c = c0 + blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= nc) return;
    int l = level[c];
    const uint64_t code = anchor[c] >> (3 * (FMM_MAXLEVEL - l));
    int o = (int)(code & 7u);
    const bool complete = ((lat >> l) & 1u) || (l <= 10 && grp[l * 8 + o] == (1u << (3 * (l - 1))));
    unsigned hm = (unsigned)(code >> 3);
    if (complete && raster && l >= 4) {
        const unsigned m = hm & 127u;
        const unsigned x = (m & 1u) | ((m >> 2) & 2u) | ((m >> 4) & 4u);
        const unsigned y = ((m >> 1) & 1u) | ((m >> 3) & 2u);
        const unsigned z = ((m >> 2) & 1u) | ((m >> 4) & 2u);
        hm = (hm & ~127u) | x | (y << 3) | (z << 5);
    }
    unsigned pos = goff[l * 8 + o] + (complete ? hm : atomicAdd(&fill[l * 8 + o], 1u));
    tgt[pos] = c;
}

__global__ void leaves_k(int nc, const int *__restrict__ nchild, unsigned *__restrict__ flag)
{
    int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c < nc) flag[c] = nchild[c] == 0;
}

__global__ void leaves_write_k(int nc, const int *__restrict__ nchild, const unsigned *__restrict__ off,
                               int *__restrict__ leaves)
{
    int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c < nc && nchild[c] == 0) leaves[off[c]] = c;
}

// leaf cell of every sorted particle: one warp per cell, leaves write their range
__global__ void pcell_k(int nc, const int *__restrict__ nchild, const int *__restrict__ begin,
                        const int *__restrict__ end, int *__restrict__ pcell)
{
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int c = (int)(t >> 5), lane = (int)(t & 31);
    if (c >= nc || nchild[c] != 0) return;
    for (int j = begin[c] + lane; j < end[c]; j += 32) pcell[j] = c;
}

// ---------------------------------------------------------------------------
// host orchestration
// ---------------------------------------------------------------------------
// number of x in [0, S) of parity par with 0 <= x + v < S
static int64_t lattice_count(int64_t S, int par, int v)
{
    const int64_t lo = std::max<int64_t>(0, -v), hi = std::min<int64_t>(S, S - v);
    if (hi <= lo) return 0;
    return (hi + 1 - par) / 2 - (lo + 1 - par) / 2;
}

// Fast path of a full octree of depth L: P2P rows from the near-field stencil,
// no pairs across levels, and the implicit same-level M2L pairs counted in
// closed form (per level, octant and stencil vector, the cells of that octant
// whose partner lies inside the lattice). Returns false (nothing done) when
// the near stencil is longer than the row sort handles.
static bool uniform_lists(fmm_ctx *h, long long K0, cudaStream_t s)
{
    const int L = h->depth, nc = h->ncells;
    const int ls = h->lvl_start[L], le = h->lvl_start[L + 1];
    const double c = h->cmac;
    // offsets beyond the lattice side never land inside it
    const int R = (int)std::min<long long>((long long)std::ceil(std::sqrt((double)K0)) + 1, (1LL << L) - 1);
    std::vector<int> nv;
    for (int vx = -R; vx <= R; vx++)
        for (int vy = -R; vy <= R; vy++)
            for (int vz = -R; vz <= R; vz++) {
                const double d2 = (double)vx * vx + (double)vy * vy + (double)vz * vz;
                if (3.0 < c * d2) continue;
                if ((int)(nv.size() / 4) == ROW_SORT_CAP) return false;  // rows too long for the row sort
                nv.insert(nv.end(), {vx, vy, vz, 0});
            }
    const int nn = (int)(nv.size() / 4);
    h->near_dev.ensure(sizeof(int) * nv.size());
    FMM_CUDA_TRY(cudaMemcpyAsync(h->near_dev.p, nv.data(), sizeof(int) * nv.size(), cudaMemcpyHostToDevice, s));
    h->p2p_ptr.ensure(sizeof(int) * (size_t)(nc + 1));
    h->row_cnt.ensure(sizeof(unsigned) * (size_t)(nc + 1));
    FMM_CUDA_TRY(cudaMemsetAsync(h->row_cnt.p, 0, sizeof(unsigned) * (size_t)(nc + 1), s));
    const unsigned nb = nblocks((int64_t)(le - ls) * 32, 256);
    near_count_k<<<nb, 256, 0, s>>>(ls, le, L, h->c_xyz.as<int4>(), h->near_dev.as<int4>(), nn, h->row_cnt.as<unsigned>());
    count_launch(h);
    scan_exclusive_u32(h, h->row_cnt.as<unsigned>(), reinterpret_cast<unsigned *>(h->p2p_ptr.as<int>()), nc + 1, nullptr, s);
    unsigned *hp = h->hpin.as<unsigned>();
    FMM_CUDA_TRY(cudaMemcpyAsync(hp, h->p2p_ptr.as<int>() + nc, sizeof(unsigned), cudaMemcpyDeviceToHost, s));
    FMM_CUDA_TRY(cudaStreamSynchronize(s));
    h->n_p2p = (int64_t)*hp;
    h->p2p_src.ensure(sizeof(int) * (size_t)std::max<int64_t>(h->n_p2p, 1));
    auto *rows = nn <= 256 ? near_rows_k<8> : nn <= 512 ? near_rows_k<16> : near_rows_k<32>;
    rows<<<nb, 256, 0, s>>>(ls, le, L, h->c_xyz.as<int4>(), h->near_dev.as<int4>(), nn, h->p2p_ptr.as<int>(),
                            h->p2p_src.as<int>());
    count_launch(h);
    check_launch("uniform lists");
    int64_t m2l = 0;
    for (int l = 1; l <= L; l++)
        for (int o = 0; o < 8; o++)
            for (int e = h->st_off[o]; e < h->st_off[o + 1]; e++) {
                const int *v = &h->st_host[4 * (size_t)e];
                m2l += lattice_count(1LL << l, o & 1, v[0]) * lattice_count(1LL << l, (o >> 1) & 1, v[1]) *
                       lattice_count(1LL << l, (o >> 2) & 1, v[2]);
            }
    h->n_m2l_implicit = m2l;
    h->n_m2lx = 0;
    return true;
}

void tree_build(fmm_ctx *h, const void *x, const void *q, int64_t n, int dt)
{
    cudaStream_t s = h->stream;
    const int TB = 256;
    h->box.ensure(sizeof(Box));
    Box *box = h->box.as<Box>();
    h->counters.ensure(sizeof(TravCounters) + 64 + sizeof(int) * 6 * (FMM_MAXLEVEL + 1));
    h->hpin.ensure(8192);

    // 1. bounding cube, keys; 2. sort
    h->keys.ensure(sizeof(uint64_t) * n);
    h->keys2.ensure(sizeof(uint64_t) * n);
    h->idx.ensure(sizeof(int) * n);
    h->idx2.ensure(sizeof(int) * n);
    h->sort_ws.ensure(sort_ws_bytes(n));
    h->launches += morton_sort_into(x, n, dt, h->keys.as<uint64_t>(), h->idx.as<int>(), h->keys2.as<uint64_t>(),
                                    h->idx2.as<int>(), h->sort_ws.p, box, h->nsm, h->sort_polls, s);

    // 3. sorted particles
    const bool mixed = h->precision == FMM_MIXED;
    const bool need64 = !mixed || dt == FMM_F64;
    if (need64) h->xs64.ensure(sizeof(double4_32a) * n);
    if (mixed) h->xs32.ensure(sizeof(float4) * n);
    double4_32a *xs64 = need64 ? h->xs64.as<double4_32a>() : nullptr;
    float4 *xs32 = mixed ? h->xs32.as<float4>() : nullptr;
    float4 *xs32lo = nullptr;
    if (mixed && dt == FMM_F64) {
        h->xs32lo.ensure(sizeof(float4) * n);
        xs32lo = h->xs32lo.as<float4>();
    }
    h->inv.ensure(sizeof(int) * n);
    if (dt == FMM_F64)
        gather_k<double><<<nblocks(n, TB), TB, 0, s>>>((const double *)x, (const double *)q, h->idx.as<int>(), n, xs64, xs32,
                                                       xs32lo, h->inv.as<int>());
    else
        gather_k<float><<<nblocks(n, TB), TB, 0, s>>>((const float *)x, (const float *)q, h->idx.as<int>(), n, xs64, xs32,
                                                      xs32lo, h->inv.as<int>());
    count_launch(h);
    check_launch("gather");

    auto check_input = [&](int nonfinite) {
        if (nonfinite) throw Error{FMM_ENONFINITE, "fmm_build: a position is NaN or infinite"};
    };
    // 4. cells
    // all cell arrays grow together; c_level's capacity stands for all of them
    auto grow_cells = [&](int need, int used) {
        size_t have = h->c_level.cap / sizeof(int);
        if (have >= (size_t)need) return;
        size_t want = std::max<size_t>((size_t)need, std::min<size_t>(2 * have, 0x7fffffff));
        h->c_level.ensure_keep(sizeof(int) * want, sizeof(int) * used, s);
        h->c_anchor.ensure_keep(sizeof(uint64_t) * want, sizeof(uint64_t) * used, s);
        h->c_begin.ensure_keep(sizeof(int) * want, sizeof(int) * used, s);
        h->c_end.ensure_keep(sizeof(int) * want, sizeof(int) * used, s);
        h->c_child.ensure_keep(sizeof(int) * want, sizeof(int) * used, s);
        h->c_nchild.ensure_keep(sizeof(int) * want, sizeof(int) * used, s);
        h->c_parent.ensure_keep(sizeof(int) * want, sizeof(int) * used, s);
        h->c_xyz.ensure_keep(sizeof(int4) * want, sizeof(int4) * used, s);
    };
    constexpr int NE = 3 * (FMM_MAXLEVEL + 1);
    auto set_extents = [&](const int *hext) {
        int E = 0;
        h->lvl_ext.assign(FMM_MAXLEVEL + 1, -1);
        for (int l = 0; l <= h->depth; l++)
            for (int d = 0; d < 3; d++)
                if (hext[NE + 3 * l + d] >= hext[3 * l + d])
                    h->lvl_ext[l] = std::max(h->lvl_ext[l], hext[NE + 3 * l + d] - hext[3 * l + d]);
        for (int l = 0; l <= h->depth; l++) E = std::max(E, h->lvl_ext[l]);
        h->lattice_extent = E;
    };
    int ncells = 1, depth = 0;
    const int64_t most = 1 + 8LL * FMM_MAXLEVEL * (n / ((int64_t)h->ncrit + 1));
    bool small = n <= TREE_SMALL_N && most <= TREE_SMALL_CELLS;
    if (small) {
        grow_cells((int)most, 0);
        h->leaves.ensure(sizeof(int) * (size_t)most);
        h->pcell.ensure(sizeof(int) * (size_t)n);
        h->small_tree.ensure(sizeof(SmallTree));
        tree_small_k<<<1, TS_T, 0, s>>>((int)n, h->ncrit, (int)most, h->keys.as<uint64_t>(), box,
                                       h->c_level.as<int>(),
                                       h->c_anchor.as<uint64_t>(), h->c_begin.as<int>(), h->c_end.as<int>(),
                                       h->c_child.as<int>(), h->c_nchild.as<int>(), h->c_parent.as<int>(),
                                       h->c_xyz.as<int4>(), h->leaves.as<int>(), h->pcell.as<int>(),
                                       h->small_tree.as<SmallTree>());
        count_launch(h);
        check_launch("small tree");
        SmallTree *st = h->hpin.as<SmallTree>();
        FMM_CUDA_TRY(cudaMemcpyAsync(st, h->small_tree.p, sizeof(SmallTree), cudaMemcpyDeviceToHost, s));
        FMM_CUDA_TRY(cudaStreamSynchronize(s));
        check_input(st->nonfinite);
        small = !st->overflow;
        if (small) {
            ncells = st->ncells;
            depth = st->depth;
            h->lvl_start.assign(st->lvl_start, st->lvl_start + depth + 2);
            h->ncells = ncells;
            h->depth = depth;
            h->nleaves = st->nleaves;
            set_extents(st->ext);
        }
    }
    if (!small) {
        // (non-finite input is reported before any further work)
        {
            int *hp = h->hpin.as<int>();
            FMM_CUDA_TRY(cudaMemcpyAsync(hp, &box->nonfinite, sizeof(int), cudaMemcpyDeviceToHost, s));
            FMM_CUDA_TRY(cudaStreamSynchronize(s));
            check_input(*hp);
        }

        const int cap = (int)std::min<int64_t>(std::max<int64_t>(1024, 2 * (n / std::max(1, h->ncrit)) + 64), 0x7fffffff);
        grow_cells(cap, 0);
        root_k<<<1, 1, 0, s>>>((int)n, h->c_level.as<int>(), h->c_anchor.as<uint64_t>(), h->c_begin.as<int>(),
                               h->c_end.as<int>(), h->c_child.as<int>(), h->c_nchild.as<int>(), h->c_parent.as<int>(),
                               h->c_xyz.as<int4>());
        count_launch(h);
        h->lvl_start.assign(1, 0);
        h->lvl_start.push_back(1);
        ncells = 1;
        depth = 0;
        for (int l = 0; l < FMM_MAXLEVEL; l++) {
            const int ls = h->lvl_start[l], le = h->lvl_start[l + 1];
            const int m = le - ls;
            if (m == 0) break;
            h->split_cnt.ensure(sizeof(unsigned) * (m + 1));
            h->split_off.ensure(sizeof(unsigned) * (m + 1));
            h->split_bnd.ensure(sizeof(int) * 9 * (size_t)m);
            split_count_k<<<nblocks((int64_t)m * 8, TB), TB, 0, s>>>(ls, le, l, h->ncrit, h->keys.as<uint64_t>(), h->c_begin.as<int>(),
                                                        h->c_end.as<int>(), h->split_cnt.as<unsigned>(), h->split_bnd.as<int>());
            count_launch(h);
            unsigned *tot = reinterpret_cast<unsigned *>(h->counters.as<char>() + sizeof(TravCounters));
            scan_exclusive_u32(h, h->split_cnt.as<unsigned>(), h->split_off.as<unsigned>(), m, tot, s);
            unsigned *hp = h->hpin.as<unsigned>();
            FMM_CUDA_TRY(cudaMemcpyAsync(hp, tot, sizeof(unsigned), cudaMemcpyDeviceToHost, s));
            FMM_CUDA_TRY(cudaStreamSynchronize(s));
            const int nnew = (int)*hp;
            if ((int64_t)le + nnew > 0x7fffffffLL) throw Error{FMM_ENOMEM, "fmm_build: too many cells"};
            grow_cells(le + nnew, le);
            split_write_k<<<nblocks(m, TB), TB, 0, s>>>(ls, le, l, h->split_cnt.as<unsigned>(), h->split_off.as<unsigned>(),
                                                        h->split_bnd.as<int>(), h->c_level.as<int>(), h->c_anchor.as<uint64_t>(),
                                                        h->c_begin.as<int>(), h->c_end.as<int>(), h->c_child.as<int>(),
                                                        h->c_nchild.as<int>(), h->c_parent.as<int>(), h->c_xyz.as<int4>());
            count_launch(h);
            check_launch("cells");
            if (nnew == 0) break;
            h->lvl_start.push_back(le + nnew);
            ncells = le + nnew;
            depth = l + 1;
        }
        h->ncells = ncells;
        h->depth = depth;
        while ((int)h->lvl_start.size() < depth + 2) h->lvl_start.push_back(ncells);
        h->lvl_start.resize(depth + 2);

        // leaves
        {
            h->leaves.ensure(sizeof(int) * ncells);
            h->split_cnt.ensure(sizeof(unsigned) * (ncells + 1));
            h->split_off.ensure(sizeof(unsigned) * (ncells + 1));
            leaves_k<<<nblocks(ncells, TB), TB, 0, s>>>(ncells, h->c_nchild.as<int>(), h->split_cnt.as<unsigned>());
            count_launch(h);
            unsigned *tot = reinterpret_cast<unsigned *>(h->counters.as<char>() + sizeof(TravCounters));
            scan_exclusive_u32(h, h->split_cnt.as<unsigned>(), h->split_off.as<unsigned>(), ncells, tot, s);
            leaves_write_k<<<nblocks(ncells, TB), TB, 0, s>>>(ncells, h->c_nchild.as<int>(), h->split_off.as<unsigned>(),
                                                              h->leaves.as<int>());
            count_launch(h);
            h->pcell.ensure(sizeof(int) * (size_t)std::max<int64_t>(n, 1));
            pcell_k<<<nblocks((int64_t)ncells * 32, TB), TB, 0, s>>>(ncells, h->c_nchild.as<int>(), h->c_begin.as<int>(),
                                                                   h->c_end.as<int>(), h->pcell.as<int>());
            count_launch(h);
            // lattice extent of the cells of every level: no same-level pair is
            // farther apart, which bounds the M2L stencil on deep adaptive trees
            int *ext = reinterpret_cast<int *>(h->counters.as<char>() + sizeof(TravCounters) + 64);
            FMM_CUDA_TRY(cudaMemsetAsync(ext, 0x7f, sizeof(int) * NE, s));
            FMM_CUDA_TRY(cudaMemsetAsync(ext + NE, 0xff, sizeof(int) * NE, s));
            extent_k<<<nblocks(ncells, TB), TB, 0, s>>>(ncells, h->c_xyz.as<int4>(), ext);
            count_launch(h);
            unsigned *hp = h->hpin.as<unsigned>();
            int *hext = reinterpret_cast<int *>(h->hpin.as<char>() + 4096);
            FMM_CUDA_TRY(cudaMemcpyAsync(hp, tot, sizeof(unsigned), cudaMemcpyDeviceToHost, s));
            FMM_CUDA_TRY(cudaMemcpyAsync(hext, ext, sizeof(int) * 2 * NE, cudaMemcpyDeviceToHost, s));
            FMM_CUDA_TRY(cudaStreamSynchronize(s));
            h->nleaves = (int)*hp;
            set_extents(hext);
        }
    }

    // 5. dual traversal
    stencil_update(h);
    stencil_levels(h, s);
    long long K0 = (long long)std::ceil(3.0 / h->cmac);
    while (K0 > 0 && 3.0 < h->cmac * (double)(K0 - 1)) K0--;
    while (!(3.0 < h->cmac * (double)K0)) K0++;
    // a full octree (all leaves on the deepest level, every level full) takes
    // the lattice stencils instead of the traversal
    bool full = h->uniform_req && depth >= 1 && depth <= 9 && h->nleaves == (1 << (3 * depth)) &&
                (int64_t)ncells == (((int64_t)1 << (3 * (depth + 1))) - 1) / 7;
    if (full) full = uniform_lists(h, K0, s);
    h->uniform_used = full;
    if (!full) {
        // the near-field stencil size bounds the P2P list of a leaf in a uniform tree
        const size_t per = (size_t)h->p2p_cap_hint + 8;
        size_t cap_p2p = std::max<size_t>(1024, std::min((size_t)h->nleaves * per, (size_t)h->nleaves * h->nleaves));
        size_t cap_m2lx = std::max<size_t>(1024, (size_t)ncells * 4);
        size_t cap_next = std::max<size_t>(1024, std::min((size_t)ncells * per, (size_t)ncells * ncells));
        h->p2p_pairs.ensure(sizeof(int2) * cap_p2p);
        h->m2lx_pairs.ensure(sizeof(int2) * cap_m2lx);
        h->frontA.ensure(sizeof(int2) * cap_next);
        h->frontB.ensure(sizeof(int2) * cap_next);
        cap_p2p = h->p2p_pairs.cap / sizeof(int2);
        cap_m2lx = h->m2lx_pairs.cap / sizeof(int2);
        TravCounters *dc = h->counters.as<TravCounters>();
        TravCounters hc = {0, 0, 0, 0};
        TravCounters *hp = h->hpin.as<TravCounters>();
        int64_t nF = 0;
        if (ncells == 1) {
            // the root is a leaf: one self pair
            int2 rp = make_int2(0, 0);
            FMM_CUDA_TRY(cudaMemcpyAsync(h->p2p_pairs.p, &rp, sizeof(int2), cudaMemcpyHostToDevice, s));
            FMM_CUDA_TRY(cudaStreamSynchronize(s));
            hc.n_p2p = 1;
        } else {
            int2 rp = make_int2(0, 0);
            FMM_CUDA_TRY(cudaMemcpyAsync(h->frontA.p, &rp, sizeof(int2), cudaMemcpyHostToDevice, s));
            FMM_CUDA_TRY(cudaStreamSynchronize(s));
            nF = 1;
        }
        while (nF > 0) {
            if (nF > 0x7fffffffLL) throw Error{FMM_ENOMEM, "fmm_build: traversal frontier too large"};
            for (int attempt = 0; attempt < 8; attempt++) {
                TravCounters start = hc;
                start.n_next = 0;
                *hp = start;
                FMM_CUDA_TRY(cudaMemcpyAsync(dc, hp, sizeof(TravCounters), cudaMemcpyHostToDevice, s));
                size_t cn = h->frontB.cap / sizeof(int2);
                expand_k<<<nblocks(nF * 8, EXPAND_T), EXPAND_T, 0, s>>>(h->frontA.as<int2>(), (unsigned)nF, h->c_xyz.as<int4>(),
                                                          h->c_child.as<int>(), h->c_nchild.as<int>(), h->cmac, K0,
                                                          h->p2p_pairs.as<int2>(), cap_p2p, h->m2lx_pairs.as<int2>(),
                                                          cap_m2lx, h->frontB.as<int2>(), cn, dc);
                count_launch(h);
                check_launch("traversal");
                FMM_CUDA_TRY(cudaMemcpyAsync(hp, dc, sizeof(TravCounters), cudaMemcpyDeviceToHost, s));
                FMM_CUDA_TRY(cudaStreamSynchronize(s));
                TravCounters got = *hp;
                bool over = false;
                if (got.n_p2p > cap_p2p) {
                    h->p2p_pairs.ensure_keep(sizeof(int2) * (size_t)(got.n_p2p * 5 / 4 + 1024), sizeof(int2) * start.n_p2p, s);
                    cap_p2p = h->p2p_pairs.cap / sizeof(int2);
                    over = true;
                }
                if (got.n_m2lx > cap_m2lx) {
                    h->m2lx_pairs.ensure_keep(sizeof(int2) * (size_t)(got.n_m2lx * 5 / 4 + 1024), sizeof(int2) * start.n_m2lx, s);
                    cap_m2lx = h->m2lx_pairs.cap / sizeof(int2);
                    over = true;
                }
                if (got.n_next > cn) {
                    h->frontB.ensure(sizeof(int2) * (size_t)(got.n_next * 5 / 4 + 1024));
                    over = true;
                }
                if (!over) {
                    hc = got;
                    break;
                }
                if (attempt == 7) throw Error{FMM_ENOMEM, "fmm_build: traversal buffers keep overflowing"};
            }
            nF = (int64_t)hc.n_next;
            std::swap(h->frontA, h->frontB);
            if (h->frontB.cap < h->frontA.cap) h->frontB.ensure(h->frontA.cap);
        }
        h->n_p2p = (int64_t)hc.n_p2p;
        h->n_m2lx = (int64_t)hc.n_m2lx;
        h->n_m2l_implicit = (int64_t)hc.n_m2l_implicit;
        if (h->n_p2p > 0x7fffffffLL || h->n_m2lx > 0x7fffffffLL)
            throw Error{FMM_ENOMEM, "fmm_build: interaction lists exceed 2^31 entries"};
        h->p2p_cap_hint = (int)std::max<int64_t>(h->p2p_cap_hint, h->n_p2p / std::max(1, h->nleaves) + 1);
    }

    // 6. CSR lists
    if (!full) pairs_to_csr(h, h->p2p_pairs.as<int2>(), h->n_p2p, h->p2p_ptr, h->p2p_src, s);
    pairs_to_csr(h, h->m2lx_pairs.as<int2>(), h->n_m2lx, h->m2lx_ptr, h->m2lx_src, s);
    h->p2p_runs.ensure(sizeof(int2) * (size_t)std::max<int64_t>(h->n_p2p, 1));
    h->p2p_nrun.ensure(sizeof(int) * (size_t)ncells);
    p2p_prepare(h, s);
    {
        unsigned long long *acc = reinterpret_cast<unsigned long long *>(h->counters.as<char>() + sizeof(TravCounters) + 8);
        FMM_CUDA_TRY(cudaMemsetAsync(acc, 0, 8, s));
        if (h->nleaves > 0) {
            p2p_runs_k<<<nblocks(h->nleaves, RUN_WARPS), 32 * RUN_WARPS, 0, s>>>(
                h->nleaves, h->leaves.as<int>(), h->p2p_ptr.as<int>(), h->p2p_src.as<int>(), h->c_begin.as<int>(),
                h->c_end.as<int>(), h->pr_ready ? h->pr_pad.as<unsigned>() : nullptr, h->pr_flag.as<unsigned>(),
                h->p2p_runs.as<int2>(), h->p2p_nrun.as<int>(), acc);
            count_launch(h);
            check_launch("p2p runs");
        }
        unsigned long long *hp = h->hpin.as<unsigned long long>();
        FMM_CUDA_TRY(cudaMemcpyAsync(hp, acc, 8, cudaMemcpyDeviceToHost, s));
        FMM_CUDA_TRY(cudaStreamSynchronize(s));
        h->n_interactions = (int64_t)*hp - n;
    }

    // 7. per-level lattice maps
    {
        std::vector<LevelDesc> ld(FMM_MAXLEVEL + 1);
        long long pool = 0;
        for (int l = 0; l <= FMM_MAXLEVEL; l++) {
            ld[l].start = l <= depth ? h->lvl_start[l] : ncells;
            ld[l].end = l <= depth ? h->lvl_start[l + 1] : ncells;
            ld[l].map_off = -1;
            ld[l].up = 0;
            if (l >= 2 && l <= depth && l <= FMM_DENSE_MAP_MAXLEVEL) {
                ld[l].map_off = pool;
                pool += 1LL << (3 * l);
            }
        }
        // deeper levels: bricks below the cells of the last dense level, while
        // all of them together are no larger than its map (64 MB). A lookup is two
        // reads of known addresses, which the tensor-core M2L has in flight ahead
        // of use; a search of a table stalls its thread until it ends. N = 1e6
        // Plummer, whose levels 9 and 10 hold half of the cells: M2L 8.2 -> 7.6 ms.
        const int top = FMM_DENSE_MAP_MAXLEVEL;
        const long long dense_end = pool;
        for (int l = top + 1; l <= depth; l++) {
            if (l - top > top) break;  // (8^top positions a brick, the limit)
            const long long words = (long long)(ld[top].end - ld[top].start) << (3 * (l - top));
            if (pool - dense_end + words > 1LL << (3 * top)) break;
            ld[l].map_off = pool;
            ld[l].up = l - top;
            ld[l].top_off = ld[top].map_off;
            ld[l].top_start = ld[top].start;
            pool += words;
        }
        h->map_pool.ensure(sizeof(int) * (size_t)std::max<long long>(pool, 1));
        if (pool > 0) FMM_CUDA_TRY(cudaMemsetAsync(h->map_pool.p, 0xff, sizeof(int) * (size_t)pool, s));
        for (int l = 2; l <= depth && l <= FMM_DENSE_MAP_MAXLEVEL; l++) {
            int m = ld[l].end - ld[l].start;
            if (m == 0) continue;
            map_fill_k<<<nblocks(m, TB), TB, 0, s>>>(ld[l].start, ld[l].end, l, h->c_anchor.as<uint64_t>(),
                                                     h->map_pool.as<int>() + ld[l].map_off);
            count_launch(h);
        }
        for (int l = top + 1; l <= depth && ld[l].map_off >= 0; l++) {
            const int m = ld[l].end - ld[l].start;
            if (m == 0) continue;
            brick_fill_k<<<nblocks(m, TB), TB, 0, s>>>(ld[l].start, ld[l].end, l, ld[l].up, ld[l].top_start,
                                                       h->c_anchor.as<uint64_t>(), h->map_pool.as<int>() + ld[l].top_off,
                                                       h->map_pool.as<int>() + ld[l].map_off);
            count_launch(h);
        }
        // the levels left: hash tables of at least twice their cells
        std::vector<long long> hoff(FMM_MAXLEVEL + 1, -1);
        long long hpool = 0;
        for (int l = FMM_DENSE_MAP_MAXLEVEL + 1; l <= depth; l++) {
            const long long m = ld[l].end - ld[l].start;
            ld[l].hash = nullptr;
            ld[l].hash_mask = 0;
            if (m == 0 || ld[l].map_off >= 0) continue;
            long long t = 64;
            while (t < 2 * m) t <<= 1;
            hoff[l] = hpool;
            ld[l].hash_mask = (unsigned)(t - 1);
            hpool += t;
        }
        if (hpool > 0) {
            h->hash_pool.ensure(sizeof(HashSlot) * (size_t)hpool);
            FMM_CUDA_TRY(cudaMemsetAsync(h->hash_pool.p, 0, sizeof(HashSlot) * (size_t)hpool, s));
            for (int l = FMM_DENSE_MAP_MAXLEVEL + 1; l <= depth; l++) {
                if (hoff[l] < 0) continue;
                HashSlot *tab = h->hash_pool.as<HashSlot>() + hoff[l];
                ld[l].hash = tab;
                const int m = ld[l].end - ld[l].start;
                hash_fill_k<<<nblocks(m, TB), TB, 0, s>>>(ld[l].start, ld[l].end, l, h->c_anchor.as<uint64_t>(), tab,
                                                          ld[l].hash_mask);
                count_launch(h);
            }
        }
        h->lvl_desc.ensure(sizeof(LevelDesc) * ld.size());
        LevelDesc *hp = reinterpret_cast<LevelDesc *>(h->hpin.as<char>() + 1024);
        std::copy(ld.begin(), ld.end(), hp);
        FMM_CUDA_TRY(cudaMemcpyAsync(h->lvl_desc.p, hp, sizeof(LevelDesc) * ld.size(), cudaMemcpyHostToDevice, s));
        check_launch("maps");
    }

    // 8. M2L target tiles: cells of levels >= 2 grouped by (level, octant)
    {
        const int tile = m2l_tile_size(h);
        const int c0 = depth >= 2 ? h->lvl_start[2] : ncells;
        const int nt = ncells - c0;
        const int pool_max = h->m2l_pool >= 0 ? h->m2l_pool : 4 * tile;
        lattice_select(h, pool_max);
        // pooled levels: one run of tiles; lattice levels: all positions;
        // complete levels: equal octant groups; others: up to one partial
        // tile per octant more
        int pooled = 0;
        int64_t ntgt = 0;
        h->ntiles_max = 0;
        for (int l = 2; l <= depth; l++) {
            const int cells = h->lvl_start[(size_t)l + 1] - h->lvl_start[(size_t)l];
            const bool lat = (h->lat_levels >> l) & 1u;
            ntgt += lat ? 1LL << (3 * l) : cells;
            if (cells <= pool_max) pooled += cells;
            else if (lat) h->ntiles_max += (1 << (3 * l)) / tile;
            else if (l <= 10 && cells == (1 << (3 * l))) h->ntiles_max += 8 * ((cells / 8 + tile - 1) / tile);
            else h->ntiles_max += cells / tile + 8;
        }
        h->ntiles_max += (pooled + tile - 1) / tile;
        h->m2l_tgt.ensure(sizeof(int) * (size_t)std::max<int64_t>(ntgt, 1));
        // positions of lattice levels without a cell
        if (ntgt > nt) FMM_CUDA_TRY(cudaMemsetAsync(h->m2l_tgt.p, 0xff, sizeof(int) * (size_t)ntgt, s));
        h->m2l_tiles.ensure(sizeof(M2LTile) * (size_t)std::max(h->ntiles_max, 1));
        h->m2l_misc.ensure(sizeof(unsigned) * 3 * 8 * (FMM_MAXLEVEL + 1) + 64);
        unsigned *grp = h->m2l_misc.as<unsigned>();
        unsigned *goff = grp + 8 * (FMM_MAXLEVEL + 1);
        unsigned *fill = goff + 8 * (FMM_MAXLEVEL + 1);
        int *ntiles = reinterpret_cast<int *>(fill + 8 * (FMM_MAXLEVEL + 1));
        FMM_CUDA_TRY(cudaMemsetAsync(grp, 0, sizeof(unsigned) * 3 * 8 * (FMM_MAXLEVEL + 1) + 64, s));
        if (nt > 0) {
            oct_count_k<<<nblocks(nt, TB), TB, 0, s>>>(c0, ncells, h->c_level.as<int>(), h->c_anchor.as<uint64_t>(), grp);
            count_launch(h);
        }
        tiles_k<<<1, 1, 0, s>>>(depth, tile, pool_max, h->lat_levels, grp, goff, h->m2l_tiles.as<M2LTile>(), ntiles);
        count_launch(h);
        if (nt > 0) {
            oct_scatter_k<<<nblocks(nt, TB), TB, 0, s>>>(c0, ncells, h->c_level.as<int>(), h->c_anchor.as<uint64_t>(),
                                                         grp, goff, fill, tile == 128 ? 1 : 0, h->lat_levels, h->m2l_tgt.as<int>());
            count_launch(h);
        }
        check_launch("m2l tiles");
        lattice_prepare(h, s);
        m2l_plan(h);
        rotation_plan(h);
    }
}

int64_t tree_m2l_total(fmm_ctx *h) { return h->n_m2l_implicit + h->n_m2lx; }

// ---------------------------------------------------------------------------
// export (tests): the implicit same-level M2L pairs are enumerated from the
// stencil and merged with the explicit ones
// ---------------------------------------------------------------------------
__global__ void stencil_pairs_k(int c0, int nc, const int *__restrict__ level, const int4 *__restrict__ xyz,
                                const uint64_t *__restrict__ anchor, const LevelDesc *__restrict__ ld,
                                const int *__restrict__ map_pool, const int4 *__restrict__ st, const int *__restrict__ st_off,
                                unsigned *__restrict__ cnt, const unsigned *__restrict__ off, int2 *__restrict__ out)
{
    int c = c0 + blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= nc) return;
    const int l = level[c];
    const int4 a = xyz[c];
    const int sh = FMM_MAXLEVEL - l;
    const int px = a.x >> sh, py = a.y >> sh, pz = a.z >> sh;
    const int o = (px & 1) | ((py & 1) << 1) | ((pz & 1) << 2);
    const LevelDesc L = ld[l];
    unsigned k = 0;
    unsigned base = off ? off[c - c0] : 0;
    for (int e = st_off[o]; e < st_off[o + 1]; e++) {
        int4 v = st[e];
        int b = level_lookup(L, map_pool, anchor, l, px + v.x, py + v.y, pz + v.z);
        if (b < 0) continue;
        if (out) out[base + k] = make_int2(c, b);
        k++;
    }
    if (!out) cnt[c - c0] = k;
}

void tree_export(fmm_ctx *h, uint64_t *keys, int32_t *perm, int32_t *level, uint64_t *anchor, int32_t *begin,
                 int32_t *end, int32_t *child, int32_t *nchild, int32_t *parent, int64_t *p2p_ptr, int32_t *p2p_idx,
                 int64_t *m2l_ptr, int32_t *m2l_idx, double *box)
{
    cudaStream_t s = h->stream;
    const int nc = h->ncells;
    const int64_t n = h->n;
    auto d2h = [&](void *dst, const void *src, size_t bytes) {
        if (dst && bytes) FMM_CUDA_TRY(cudaMemcpyAsync(dst, src, bytes, cudaMemcpyDeviceToHost, s));
    };
    d2h(keys, h->keys.p, sizeof(uint64_t) * n);
    d2h(perm, h->idx.p, sizeof(int) * n);
    d2h(level, h->c_level.p, sizeof(int) * nc);
    d2h(anchor, h->c_anchor.p, sizeof(uint64_t) * nc);
    d2h(begin, h->c_begin.p, sizeof(int) * nc);
    d2h(end, h->c_end.p, sizeof(int) * nc);
    d2h(child, h->c_child.p, sizeof(int) * nc);
    d2h(nchild, h->c_nchild.p, sizeof(int) * nc);
    d2h(parent, h->c_parent.p, sizeof(int) * nc);
    if (box) {
        Box hb;
        FMM_CUDA_TRY(cudaMemcpyAsync(&hb, h->box.p, sizeof(Box), cudaMemcpyDeviceToHost, s));
        FMM_CUDA_TRY(cudaStreamSynchronize(s));
        box[0] = hb.origin[0];
        box[1] = hb.origin[1];
        box[2] = hb.origin[2];
        box[3] = hb.R0;
    }
    if (p2p_ptr || p2p_idx) {
        std::vector<int> ptr(nc + 1);
        FMM_CUDA_TRY(cudaMemcpyAsync(ptr.data(), h->p2p_ptr.p, sizeof(int) * (nc + 1), cudaMemcpyDeviceToHost, s));
        d2h(p2p_idx, h->p2p_src.p, sizeof(int) * h->n_p2p);
        FMM_CUDA_TRY(cudaStreamSynchronize(s));
        if (p2p_ptr)
            for (int i = 0; i <= nc; i++) p2p_ptr[i] = ptr[i];
    }
    if (m2l_ptr || m2l_idx) {
        // implicit same-level pairs: count, scan, write
        const int c0 = h->depth >= 2 ? h->lvl_start[2] : nc;
        const int m = nc - c0;
        int64_t nimp = 0;
        DevBuf cnt, off, pairs, ptr, src;
        if (m > 0) {
            cnt.ensure(sizeof(unsigned) * (m + 1));
            off.ensure(sizeof(unsigned) * (m + 1));
            const int *st_off = stencil_offsets(h);
            stencil_pairs_k<<<nblocks(m, 128), 128, 0, s>>>(c0, nc, h->c_level.as<int>(), h->c_xyz.as<int4>(),
                                                            h->c_anchor.as<uint64_t>(), h->lvl_desc.as<LevelDesc>(),
                                                            h->map_pool.as<int>(), h->st_dev.as<int4>(), st_off,
                                                            cnt.as<unsigned>(), nullptr, nullptr);
            count_launch(h);
            unsigned *tot = reinterpret_cast<unsigned *>(h->counters.as<char>() + sizeof(TravCounters));
            scan_exclusive_u32(h, cnt.as<unsigned>(), off.as<unsigned>(), m, tot, s);
            unsigned ht = 0;
            FMM_CUDA_TRY(cudaMemcpyAsync(&ht, tot, sizeof(unsigned), cudaMemcpyDeviceToHost, s));
            FMM_CUDA_TRY(cudaStreamSynchronize(s));
            nimp = ht;
        }
        const int64_t ntot = nimp + h->n_m2lx;
        pairs.ensure(sizeof(int2) * (size_t)std::max<int64_t>(ntot, 1));
        if (m > 0 && nimp > 0) {
            const int *st_off = stencil_offsets(h);
            stencil_pairs_k<<<nblocks(m, 128), 128, 0, s>>>(c0, nc, h->c_level.as<int>(), h->c_xyz.as<int4>(),
                                                            h->c_anchor.as<uint64_t>(), h->lvl_desc.as<LevelDesc>(),
                                                            h->map_pool.as<int>(), h->st_dev.as<int4>(), st_off,
                                                            cnt.as<unsigned>(), off.as<unsigned>(), pairs.as<int2>());
            count_launch(h);
        }
        if (h->n_m2lx > 0)
            FMM_CUDA_TRY(cudaMemcpyAsync(pairs.as<int2>() + nimp, h->m2lx_pairs.p, sizeof(int2) * h->n_m2lx,
                                         cudaMemcpyDeviceToDevice, s));
        pairs_to_csr(h, pairs.as<int2>(), ntot, ptr, src, s);
        std::vector<int> hptr(nc + 1);
        FMM_CUDA_TRY(cudaMemcpyAsync(hptr.data(), ptr.p, sizeof(int) * (nc + 1), cudaMemcpyDeviceToHost, s));
        d2h(m2l_idx, src.p, sizeof(int) * ntot);
        FMM_CUDA_TRY(cudaStreamSynchronize(s));
        if (m2l_ptr)
            for (int i = 0; i <= nc; i++) m2l_ptr[i] = hptr[i];
        cnt.release();
        off.release();
        pairs.release();
        ptr.release();
        src.release();
    }
    FMM_CUDA_TRY(cudaStreamSynchronize(s));
}

}  // namespace fmm
