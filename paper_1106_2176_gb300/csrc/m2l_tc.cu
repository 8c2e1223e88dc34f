// M2L on the tensor cores (tcgen05, sm_103a).
//
// Same-level M2L (Sec. 2.1 of Yokota & Barba, arXiv:1106.2176) is a dense
// contraction once the expansions are scaled by their cell width: for a tile
// of 128 target cells of one level and one octant and a translation vector v
// of the octant's stencil,
//     L~[128 x p^2] += gather_v(M~)[128 x p^2] * T_v^T,
// T_v the level-independent p^2 x p^2 real operator. Sec. 5 notes that M2L at
// all levels needs no synchronisation between levels: one launch covers every
// level's tiles.
//
// Precision: A = M~ and B = T_v are split into two FP16 values each, hi and
// lo = x - hi (both rounded to nearest: 22 bits, an error below 2^-23 of x),
// and the MMAs compute A_hi [T_hi ; T_lo] plus A_lo T_hi, accumulating in
// FP32 in tensor memory: the main sum in columns [0, NP), the small
// correction terms in [NP, 2 NP). FP16's 11-bit significand is TF32's, at
// twice the MMA rate and half the operand bytes; what it lacks is exponent
// range, so the operands are brought into range by powers of two (exact):
//   - coefficient (n, m) of M~ is multiplied and that of L~ divided by
//     2^round(log2 sqrt((n+m)! (n-m)!)), which takes the factorials out of the
//     solid harmonics; the powers of the distance in T are then balanced by
//     2^-n on M~ and one power of two per degree of L~, so that the largest
//     entries of every degree's rows lie in [2^13, 2^14);
//   - a level's rows are multiplied by 2^e so that the largest coefficient of
//     the level lies in [2^14, 2^15) (e from a maximum taken each evaluation).
// FP16's subnormals end 2^-39 below that maximum: a cell far below its level's
// largest keeps fewer bits than FP32. Where that may show, at targets all of
// whose surroundings are 2^-16 below (weak charges far from strong ones that
// cancel: m2l_exposed), the level is "wide" and its tiles are summed in FP32 on
// the CUDA cores (m2l_wide_tile). Every GV vectors an accumulator is drained into
// per-thread FP32 (hi, lo) TwoSum registers.
//
// Per CTA (two groups of 4 worker warps, NM MMA warps and NM producer warps) a
// ring of NS stages, one unit (vector v, k-block of 64
// coefficients) each: 128 rows of A_hi and A_lo and the operator block
// [T_hi ; T_lo], all 128B-swizzled in shared memory, where the MMAs read both
// operands.
//   - a producer brings the unit's operator block with one bulk copy and, on
//     complete and nearly complete levels (lattice tiles), A_hi and A_lo with
//     one TMA tile load each; the workers then only drain.
//   - on other levels the worker group u % 2 gathers the unit's rows with
//     cp.async straight into the stage (sources found by lattice lookups
//     fetched ahead into a ring; zero fill where a cell is absent). The
//     copies' completion arrives on the stage's mbarrier; the MMA thread
//     orders them before its asynchronous reads with a proxy fence.
//   - an MMA warp issues the tcgen05.mma of a vector's units into its
//     accumulators and commits each unit to its stage's "empty" barrier. With
//     one warp and NP <= 64 the tensor pipe idles while that warp waits for the
//     next stage and commits (about 750 of 1,260 cycles per vector at p = 8):
//     there two MMA warps and two producers take every other vector each, in
//     stages of their own parity.
// The rows are split into FP16 once per evaluation (m2l_split_k) and not once
// per vector, so nothing but copies and MMAs is left per vector.
// Bound (N = 1e7, p = 8, 7.1 ms; 19.8 with TF32 pairs split per vector in
// worker warps, 12.2 with one MMA warp): the copies, 48 KB per vector and tile
// from L2 at 69 bytes per clock and SM; without the MMAs the launch takes 6.75
// ms.
// p = 9 .. 11 (60 KB stages, three of them, one MMA warp): the waits and
// commits between the units, 2.66 ms at N = 1e6, p = 10 (6.6 with TF32).
//
// A tree with few tiles (5 at N = 16,384) would leave most SMs idle: the
// vectors of every tile are then cut into nsplit ranges, one CTA each
// (m2l_plan). Each CTA writes its (hi, lo) sums and the last one of a tile to
// finish adds the ranges in order, so results do not depend on scheduling. The
// ranges start at multiples of one chunk of whole drain groups, whatever the
// length of the tile's own list: a cell's sums do not depend on the tile that
// it falls into either (cells of incomplete levels are placed in arrival order).
//
// Every wait is bounded; on a timeout the kernel records an error code and
// leaves after its copies have landed and its TMEM is released.
#include <algorithm>
#include <array>
#include <climits>
#include <cmath>
#include <cstring>
#include <map>
#include <memory>
#include <mutex>
#include <tuple>

#include <cuda.h>  // CUtensorMap and its encoding enums (the encoder comes from the runtime's driver entry point)
#include <cuda_fp16.h>

#include "fmm_internal.cuh"
#include "m2l_norm.cuh"
#include "ptx_sm100.cuh"

namespace fmm {

static inline unsigned nblk(int64_t n, int bs) { return (unsigned)((n + bs - 1) / bs); }

// ---------------------------------------------------------------------------
// tile geometry
// ---------------------------------------------------------------------------
// NP: p^2 padded to a multiple of 16 (the MMA's N). A cell's row is KB blocks
// of 64 coefficients, each 128 bytes of hi and 128 bytes of lo; with NP <= 32
// both halves fit one 128-byte row (PACK: hi in the first 64 bytes, lo in the
// last), and so do T_hi and T_lo.
// Tensor memory: two accumulator buffers of 2 NP columns (main | correction)
// for each of the NM MMA warps. Warp m takes the vectors w = NM i + m, GV of
// them to an accumulator: group (i + OFF m) / GV, so that the drains of two
// warps alternate.
// Thread (r, g) drains output columns [g HN, (g + 1) HN) of row r.
template <int NP>
struct TcCfg {
    static constexpr int M = 128;                  // target rows per tile
    static constexpr int NW = 8;                   // worker warps
    static constexpr int NG = 2;                   // worker groups
    static constexpr bool PACK = NP <= 32;
    static constexpr int KB = (NP + 63) / 64;      // k-blocks per vector
    static constexpr int ROWB = PACK ? 128 : 256;  // bytes of a row's k-block (hi and lo)
    static constexpr int A_BYTES = M * ROWB;
    static constexpr int B_BYTES = (PACK ? 1 : 2) * NP * 128;
    static constexpr int STAGE = A_BYTES + B_BYTES;
    static constexpr int QU = 7;                   // lookahead of either read of a source lookup (units of the group)
    static constexpr int RINGU = 16;               // slots, more than 2 QU
    static constexpr int RING = NG * RINGU * M * 4;
    static constexpr int BAR = 768;                // mbarriers (first 512 bytes), then the CTA's job
    static constexpr int NS_FIT = (226 * 1024 - RING - BAR - 1024) / STAGE;
    // MMA warps (and producers). Two only where a vector is one unit and the
    // stages number an even count: unit u, stage u % NS, then always meets the
    // same warps, and no wait on a stage's barrier can be two phases ahead
    // (which its parity would not tell from a completed one).
    static constexpr int NM = KB == 1 ? 2 : 1;
    static constexpr int MMA_WARP = NW, P_WARP = NW + NM;
    static constexpr int NT = 32 * (NW + 4);       // threads (with NM = 1 two warps idle)
    static constexpr int NS = NS_FIT > 6 ? 6 : NM == 2 ? NS_FIT & ~1 : NS_FIT;
    static constexpr int SMEM = NS * STAGE + RING + BAR + 1024;
    static constexpr int TCOLS = 512;
    static constexpr int AC = 2;                   // accumulator buffers per MMA warp
    static constexpr int GV = 8;                   // vectors per accumulator drain
    static constexpr int OFF = GV / 2;
    static constexpr int HN = NP / 2;              // output coefficients per thread
    // Registers: 168 a thread at launch (384 threads). The workers hold 2 HN sums
    // besides the gathers' state; from NP = 64 on they take REG_W and the other
    // four warps keep REG_O, together 63,488 of the launch's 64,512 (launch_tc
    // checks). Spills at NP = 112 (p = 10) 184 -> 8 bytes; M2L at N = 1e5, p = 10
    // 1.20 -> 0.92 ms, at N = 1e6 3.09 -> 2.66 ms. Not in the persistent kernel,
    // whose roles meet again at every item.
    static constexpr int REG_W = 216, REG_O = 64;
    static constexpr bool REGS = NP >= 64;
    // a gathering worker drains a group once it has to wait for a vector more
    // than LATE past the group's last one: the group is then finished or about
    // to be, and the next group of the same buffer has not begun
    static constexpr int LATE = (NS + KB - 1) / KB;
    static_assert(NP % 16 == 0 && STAGE % 1024 == 0 && NS >= 3 && 2 * NM * AC * NP <= TCOLS && SMEM <= 227 * 1024 &&
                      LATE < GV && 2 * QU >= NS && (NM == 1 || (KB == 1 && NS % 2 == 0)),
                  "stage budget");
};

// ---------------------------------------------------------------------------
// operand rows
// ---------------------------------------------------------------------------
// Largest |M~ a| (a: m2l_norm) of every cell and of every level from 2 on, as FP32
// bits (the order of non-negative floats), over the finite coefficients; lmax starts
// at zero. grid.y: levels from 2 on (the few cells above go with 2); a warp walks cells, lane i holds coefficients i, i + 32, ...
__global__ void __launch_bounds__(256) m2l_lmax_k(const float *__restrict__ M, int PP, const __grid_constant__ M2LLevels lv,
                                                  unsigned *__restrict__ cmax, unsigned *__restrict__ lmax)
{
    const int l = 2 + blockIdx.y, lane = threadIdx.x & 31;
    const int c1 = lv.start[l + 1];
    float a[4];
#pragma unroll
    for (int r = 0; r < 4; r++) a[r] = m2l_norm(lane + 32 * r);
    unsigned best = 0;
    constexpr int U = 4;  // cells in flight
    const int step = (int)gridDim.x * 8;
    for (int c0 = (l > 2 ? lv.start[l] : 0) + (int)(blockIdx.x * 8 + (threadIdx.x >> 5)); c0 < c1; c0 += U * step) {
        unsigned b[U];
#pragma unroll
        for (int u = 0; u < U; u++) {
            b[u] = 0;
            if (c0 + u * step >= c1) continue;
            const float *Mc = M + (size_t)(c0 + u * step) * PP;
#pragma unroll
            for (int r = 0; r < 4; r++)
                if (lane + 32 * r < PP) b[u] = max(b[u], m2l_mag(Mc[lane + 32 * r] * a[r]));
        }
#pragma unroll
        for (int u = 0; u < U; u++) {
            if (c0 + u * step >= c1) break;
            b[u] = __reduce_max_sync(0xffffffffu, b[u]);
            if (lane == 0) cmax[c0 + u * step] = b[u];
            if (c0 + u * step >= lv.start[l]) best = max(best, b[u]);
        }
    }
    __shared__ unsigned sb[8];
    if (lane == 0) sb[threadIdx.x >> 5] = best;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < 8; w++) best = max(best, sb[w]);
        if (best > *(volatile unsigned *)(lmax + l)) atomicMax(lmax + l, best);
    }
}

// coefficients 8 ch .. 8 ch + 7 of one cell as FP16 (hi, lo): M~ a 2^e
template <int NP>
__device__ __forceinline__ void m2l_split_chunk(const float *__restrict__ Mc, int PP, int ch, int e,
                                                unsigned char *__restrict__ row)
{
    using C = TcCfg<NP>;
    __align__(16) float v[8];  // (written and read as 16-byte vectors, whether in registers or in memory)
#pragma unroll
    for (int i = 0; i < 8; i++) v[i] = 0.f;
    const int k0 = 8 * ch;
    if ((PP & 3) == 0) {  // rows start on 16-byte boundaries
        if (k0 < PP) *reinterpret_cast<float4 *>(v) = *reinterpret_cast<const float4 *>(Mc + k0);
        if (k0 + 4 < PP) *reinterpret_cast<float4 *>(v + 4) = *reinterpret_cast<const float4 *>(Mc + k0 + 4);
    } else {
#pragma unroll
        for (int i = 0; i < 8; i++)
            if (k0 + i < PP) v[i] = Mc[k0 + i];
    }
    // 2^e in two factors: e may lie outside the exponent range of one float
    const float s1 = m2l_pow2(e >> 1), s2 = m2l_pow2(e - (e >> 1));
    __align__(16) __half h[8], w[8];
#pragma unroll
    for (int i = 0; i < 8; i++) {
        const float x = (v[i] * m2l_norm(k0 + i)) * s1 * s2;
        h[i] = __float2half_rn(x);
        w[i] = __float2half_rn(x - __half2float(h[i]));
    }
    const int off = C::PACK ? ch * 16 : (ch >> 3) * 256 + (ch & 7) * 16;
    *reinterpret_cast<uint4 *>(row + off) = *reinterpret_cast<const uint4 *>(h);
    *reinterpret_cast<uint4 *>(row + off + (C::PACK ? 64 : 128)) = *reinterpret_cast<const uint4 *>(w);
}

// FP16 rows of the cells from level 2 on, and the marks of wide levels. A cell of a lattice level (bit l of
// lat.levels) goes to the lattice copy of its level: the row of position (x, y,
// z) at ((b H + z/2) H + y/2) H + x/2, b = (x & 1) | (y & 1) << 1 | (z & 1) << 2
// its octant bits and H = 2^(l-1), so that the cells of one octant form an H^3
// block in x, y, z order and the sources of a block of targets under one
// translation are a shifted block. Other cells go to row c of `rows`.
template <int NP>
__global__ void __launch_bounds__(256) m2l_split_k(const float *__restrict__ M, int PP, const int4 *__restrict__ xyz, int c0,
                                                   int nc, const int *__restrict__ parent,
                                                   const unsigned *__restrict__ cmax, unsigned *ws,
                                                   const __grid_constant__ M2LLattice lat, unsigned char *__restrict__ rows,
                                                   unsigned char *__restrict__ mlat)
{
    using C = TcCfg<NP>;
    constexpr int NCH = NP / 8, RB = C::KB * C::ROWB;
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= (int64_t)(nc - c0) * NCH) return;
    const int c = c0 + (int)(i / NCH), ch = (int)(i % NCH);
    const int4 a = xyz[c];
    const int l = a.w;
    unsigned char *row = rows + (size_t)c * RB;
    if ((lat.levels >> l) & 1u) {
        const int sh = FMM_MAXLEVEL - l;
        const int64_t H = 1ll << (l - 1);
        const int x = a.x >> sh, y = a.y >> sh, z = a.z >> sh;
        const int b = (x & 1) | ((y & 1) << 1) | ((z & 1) << 2);
        row = mlat + (lat.off[l] + ((b * H + (z >> 1)) * H + (y >> 1)) * H + (x >> 1)) * RB;
    }
    m2l_split_chunk<NP>(M + (size_t)c * PP, PP, ch, m2l_exponent(ws[l]), row);
    if (ch == 0) m2l_mark(c, l, cmax, parent, ws, nullptr);
}

// bits 0, 3, 6, ... of a Morton code below 2^30
__device__ __forceinline__ uint32_t every_third(uint32_t v)
{
    v &= 0x09249249u;
    v = (v | (v >> 2)) & 0x030c30c3u;
    v = (v | (v >> 4)) & 0x0300f00fu;
    v = (v | (v >> 8)) & 0x030000ffu;
    v = (v | (v >> 16)) & 0x3ffu;
    return v;
}

// tiles of a wide level, and pooled tiles once any level is wide
__device__ __forceinline__ bool m2l_is_wide(unsigned wide, const M2LTile &t)
{
    return wide && (t.octant == 8 || ((wide >> t.level) & 1u));
}

// One (tile, range) item in FP32 on the CUDA cores, by the first 256 threads of a
// block (all of them take part in the barriers). Per vector C[row][r] += sum_c A[row][c] T[r][c]:
// A the sources' M~ a, T = (hi + lo) 2^-14 of the operator image, both staged in
// shared memory 32 coefficients at a time; thread (ty, tx) holds rows 8 ty .. 8 ty
// + 7 and columns tx, tx + 16, .... Sums run over 8 vectors in FP32, as in tensor
// memory, then into (hi, lo) pairs, and over the ranges of a tile as there. Slow
// (29 ms for 10^6 particles, p = 8, against 5.2 on the tensor cores) and rare.
constexpr int WD_T = 256, WD_KC = 32, WD_LD = 132, WD_V = 8;
template <int NP>
struct WideShared {
    float A[WD_KC][WD_LD];
    float T[WD_KC][NP];
    int src[WD_V][128];
    int any[WD_V];
    int last;
};

template <int NP>
__device__ __noinline__ void m2l_wide_tile(const M2LJob &J, int p, int item, WideShared<NP> &sh)
{
    using C = TcCfg<NP>;
    constexpr int NC = NP / 16;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, PP = p * p;
    const int tx = tid & 15, ty = (tid >> 4) & 15;
    const bool on = tid < WD_T;
    const int tile = item / J.nsplit, split = item - tile * J.nsplit;
    const M2LTile td = J.tiles[tile];
    const int nvt = J.st_off[10 + td.octant * (FMM_MAXLEVEL + 1) + td.level];
    const int w0 = (int)min((long long)nvt, (long long)split * J.chunk), w1 = (int)min((long long)nvt, (long long)w0 + J.chunk);
    const int e0 = J.st_off[td.octant] + w0, nv = w1 - w0;
    // thread t looks up sources of row t % 128
    int cell = -1, rl = td.level, px = 0, py = 0, pz = 0, ro = 0;
    if (on && (tid & 127) < td.count) cell = J.tgt[td.start + (tid & 127)];  // (-1: a lattice position without a cell)
    if (cell >= 0) {
        const int4 a = J.xyz[cell];
        rl = a.w;
        const int s = FMM_MAXLEVEL - rl;
        px = a.x >> s;
        py = a.y >> s;
        pz = a.z >> s;
        ro = (px & 1) | ((py & 1) << 1) | ((pz & 1) << 2);
    }
    float acc[8][NC], hi[8][NC], lo[8][NC];
#pragma unroll
    for (int i = 0; i < 8; i++)
#pragma unroll
        for (int j = 0; j < NC; j++) hi[i][j] = lo[i][j] = 0.f;
    for (int v0 = 0; v0 < nv; v0 += WD_V) {
        __syncthreads();  // the last group's sources are used up
        if (tid < WD_V) sh.any[tid] = 0;
        __syncthreads();
        if (on)
            for (int k = tid >> 7; k < WD_V; k += WD_T / 128) {
                int b = -1;
                if (v0 + k < nv && cell >= 0) {
                    const int4 v = J.st[e0 + v0 + k];
                    if ((v.w >> (16 + ro)) & 1) b = level_lookup(J.ld[rl], J.map_pool, J.anchor, rl, px + v.x, py + v.y, pz + v.z);
                }
                sh.src[k][tid & 127] = b;
                if (b >= 0) sh.any[k] = 1;
            }
#pragma unroll
        for (int i = 0; i < 8; i++)
#pragma unroll
            for (int j = 0; j < NC; j++) acc[i][j] = 0.f;
        __syncthreads();
        for (int k = 0; k < WD_V && v0 + k < nv; k++) {
            if (!sh.any[k]) continue;  // (the same in every thread)
            const unsigned char *op = J.ttab + (size_t)(J.st[e0 + v0 + k].w & 0xffff) * C::KB * C::B_BYTES;
            for (int c0 = 0; c0 < PP; c0 += WD_KC) {
                __syncthreads();  // the staged coefficients are used up
                if (on) {
                    const float a = c0 + lane < PP ? m2l_norm(c0 + lane) : 0.f;
                    constexpr int RW = 128 / (WD_T / 32);  // rows per warp, all loads in flight before the first store
                    float m[RW];
#pragma unroll
                    for (int i = 0; i < RW; i++) {
                        const int b = sh.src[k][warp + i * (WD_T / 32)];
                        m[i] = b >= 0 && c0 + lane < PP ? J.M[(size_t)b * PP + c0 + lane] * a : 0.f;
                    }
#pragma unroll
                    for (int i = 0; i < RW; i++) sh.A[lane][warp + i * (WD_T / 32)] = m[i];
                    // 8 coefficients of one output a thread
                    for (int i = tid; i < NP * (WD_KC / 8); i += WD_T) {
                        const int r = i % NP, q = i / NP;
                        const int ch = ((c0 & 63) >> 3) + q;  // its 16-byte chunk in the k-block's row
                        const unsigned char *blk = op + (size_t)(c0 >> 6) * C::B_BYTES;
                        const unsigned char *ph = blk + r * 128 + ((ch ^ (r & 7)) << 4);
                        const unsigned char *pl = C::PACK ? blk + r * 128 + (((ch + 4) ^ (r & 7)) << 4)
                                                          : blk + (NP + r) * 128 + ((ch ^ ((NP + r) & 7)) << 4);
                        const uint4 h4 = *reinterpret_cast<const uint4 *>(ph), l4 = *reinterpret_cast<const uint4 *>(pl);
                        const unsigned hw[4] = {h4.x, h4.y, h4.z, h4.w}, lw[4] = {l4.x, l4.y, l4.z, l4.w};
#pragma unroll
                        for (int n = 0; n < 8; n++) {
                            const unsigned short hb = (unsigned short)(hw[n / 2] >> (16 * (n & 1)));
                            const unsigned short lb = (unsigned short)(lw[n / 2] >> (16 * (n & 1)));
                            sh.T[8 * q + n][r] = (__half2float(__ushort_as_half(hb)) + __half2float(__ushort_as_half(lb))) * 0x1p-14f;
                        }
                    }
                }
                __syncthreads();
                if (on) {
                    const int kc = min(WD_KC, PP - c0);
                    for (int c = 0; c < kc; c++) {
                        float a[8], t[NC];
#pragma unroll
                        for (int i = 0; i < 8; i++) a[i] = sh.A[c][8 * ty + i];
#pragma unroll
                        for (int j = 0; j < NC; j++) t[j] = sh.T[c][tx + 16 * j];
#pragma unroll
                        for (int i = 0; i < 8; i++)
#pragma unroll
                            for (int j = 0; j < NC; j++) acc[i][j] = fmaf(a[i], t[j], acc[i][j]);
                    }
                }
            }
        }
#pragma unroll
        for (int i = 0; i < 8; i++)
#pragma unroll
            for (int j = 0; j < NC; j++) two_sum_acc(hi[i][j], lo[i][j], acc[i][j]);
    }
    auto put = [&](int row, int r, float x) {
        const int c = row < td.count ? J.tgt[td.start + row] : -1, t = J.rowexp[r] + 14;
        if (c >= 0) J.L[(size_t)c * PP + r] += (x * m2l_pow2(t >> 1)) * m2l_pow2(t - (t >> 1));
    };
    const size_t rng = (size_t)PP * 128;
    if (on)
#pragma unroll
        for (int i = 0; i < 8; i++)
#pragma unroll
            for (int j = 0; j < NC; j++) {
                const int row = 8 * ty + i, r = tx + 16 * j;
                if (r >= PP) continue;
                if (J.nsplit == 1) put(row, r, hi[i][j] + lo[i][j]);
                else __stcg(&J.part[(size_t)item * rng + (size_t)r * 128 + row], make_float2(hi[i][j], lo[i][j]));
            }
    if (J.nsplit == 1) return;
    // the tile's last range to finish adds them all in order
    __threadfence();
    __syncthreads();
    if (tid == 0) {
        sh.last = atomicAdd(&J.tcnt[tile], 1u) == (unsigned)(J.nsplit - 1);
        if (sh.last) J.tcnt[tile] = 0u;
        __threadfence();
    }
    __syncthreads();
    if (!sh.last || !on) return;
    for (int i = tid; i < PP * 128; i += WD_T) {
        float h = 0.f, w = 0.f;
        for (int k = 0; k < J.nsplit; k++) {
            const float2 v = __ldcg(&J.part[((size_t)tile * J.nsplit + k) * rng + i]);
            two_sum_acc(h, w, v.x);
            w += v.y;
        }
        put(i & 127, i >> 7, h + w);
    }
}

// the job that holds queue item `it` (the last one: also items past its end)
__device__ __forceinline__ int job_of(const M2LJob *__restrict__ jobs, int njobs, int it)
{
    int lo = 0, hi = njobs - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (jobs[mid].item0 <= it) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

template <int NP, bool PERSIST>
__global__ void __launch_bounds__(TcCfg<NP>::NT, 1)
    m2l_tc_k(int p, const __grid_constant__ M2LJob one, const M2LJob *__restrict__ jobs, int njobs,
             int *__restrict__ queue, const unsigned *__restrict__ any, int *__restrict__ err)
{
    // PERSIST (many systems: jobs[], njobs entries sorted by item0): each CTA
    // takes (tile, range) items from the queue until it is empty. Otherwise
    // CTA b computes item b of the single job `one`, read from the parameter
    // space, which measured faster for one system than the persistent loop.
    // *any: zero if no level is wide.
    using C = TcCfg<NP>;
    constexpr int NS = C::NS, NM = C::NM, QU = C::QU, RINGU = C::RINGU, KB = C::KB;
    constexpr bool PACK = C::PACK;
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char *base = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
    int *ring = reinterpret_cast<int *>(base + NS * C::STAGE);  // NG x RINGU x M
    uint64_t *bar = reinterpret_cast<uint64_t *>(reinterpret_cast<unsigned char *>(ring) + C::RING);
    uint64_t *full = bar;                     // NS: bytes of the producer's copies
    uint64_t *gfull = full + NS;              // NS: cp.async arrivals of a group's 128 threads (gathered tiles)
    uint64_t *empty = gfull + NS;             // NS: MMA commits
    uint64_t *acc_full = empty + NS;          // 2 AC: MMA commits at the end of a group of vectors
    uint64_t *acc_empty = acc_full + 2 * C::AC;  // 2 AC: one arrival per worker warp after a drain
    uint64_t *fin = acc_empty + 2 * C::AC;    // 2: last commit of each MMA warp
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(fin + 2);
    int *abort_flag = reinterpret_cast<int *>(tmem_slot + 1);
    int *s_item = abort_flag + 1;                 // this CTA's current item (-1: none left)
    int *s_last = s_item + 1;                     // this CTA finished its tile last
    int *s_wide = s_last + 1;                     // (PERSIST) *any, once per CTA
    M2LJob *s_job = reinterpret_cast<M2LJob *>(reinterpret_cast<unsigned char *>(bar) + 512);  // its job
    static_assert(sizeof(uint64_t) * (3 * NS + 4 * C::AC + 2) + 20 <= 512 && 512 + sizeof(M2LJob) <= C::BAR, "barrier area");

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    static_assert(sizeof(WideShared<NP>) <= NS * C::STAGE, "shared memory of a wide tile");
    if (PERSIST) {
        if (tid == 0) *s_wide = (int)*any;
    } else {
        const unsigned wide = *any;
        if ((int)blockIdx.x >= *one.ntiles * one.nsplit) return;
        if (wide && m2l_is_wide(wide, one.tiles[(int)blockIdx.x / one.nsplit])) {
            m2l_wide_tile<NP>(one, p, (int)blockIdx.x, *reinterpret_cast<WideShared<NP> *>(base));
            return;
        }
    }
    if (warp == C::MMA_WARP) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                     "r"(C::TCOLS));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    for (int pass = 0; PERSIST || pass == 0; pass++) {
    if (tid == 0) {
        if (PERSIST) {
            do {  // (wide tiles are left for the end)
                const int it = atomicAdd(queue, 1);
                *s_job = jobs[job_of(jobs, njobs, it)];
                const int t = it - s_job->item0;
                *s_item = (t >= 0 && t < s_job->count) ? t : -1;
            } while (*s_wide && *s_item >= 0 && m2l_is_wide(s_job->ws[M2LW_WIDE], s_job->tiles[*s_item / s_job->nsplit]));
        } else {
            *s_item = (int)blockIdx.x;
        }
        // the item's barriers start from phase 0 (the previous item left
        // every barrier idle: all its waits, copies and commits completed)
        for (int s = 0; s < NS; s++) {
            mbar_init(&full[s], 1);
            mbar_init(&gfull[s], 128);
            mbar_init(&empty[s], 1);
        }
        for (int b = 0; b < 2 * C::AC; b++) {
            mbar_init(&acc_full[b], 1);
            mbar_init(&acc_empty[b], C::NW);
        }
        mbar_init(&fin[0], 1);
        mbar_init(&fin[1], 1);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    const int item = *s_item;
    if (item < 0) break;
    const M2LJob &J = PERSIST ? *s_job : one;
    const int nsplit = J.nsplit, tile = item / nsplit, split = item - tile * nsplit;
    const M2LTile td = J.tiles[tile];
    const int PP = p * p;
    const int l = td.level;
    const int4 *__restrict__ st = J.st;
    // the set's entries are sorted by reach: only a prefix can hit a cell;
    // this CTA's range of it
    const int nvt = J.st_off[10 + td.octant * (FMM_MAXLEVEL + 1) + l];
    const int w0 = (int)min((long long)nvt, (long long)split * J.chunk), w1 = (int)min((long long)nvt, (long long)w0 + J.chunk);
    const int e0 = J.st_off[td.octant] + w0, nv = w1 - w0;
    const int nunits = nv * KB;
    // Lattice tile (a level with a lattice copy of its rows): the tile is an
    // 8 x 4 x 4 block of its octant's sub-lattice with rows in x, y, z
    // order, and for every vector the sources form the same block shifted, in
    // the sub-lattice of the source octant; positions outside the level or
    // without a cell arrive as zeros, as absent cells do.
    // (persistent launches serve the batch engine, which gathers everywhere)
    const bool lat = !PERSIST && J.lat_maps != nullptr && td.block >= 0;

    if (warp >= C::NW) {
        if constexpr (!PERSIST && C::REGS) asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(C::REG_O));
        if (warp < C::P_WARP) {
            // ----------------------------------------------------------- MMA warps
            // (the waits and commits, a few hundred cycles per unit, of one warp
            // overlap the other's MMAs). The whole warp runs the loop and one
            // elected lane issues: the branch on elect.sync lets the compiler keep
            // the descriptors in uniform registers (7.25 against 7.75 ms at
            // N = 1e7, p = 8, with one lane running the loop).
            const int m = warp - C::MMA_WARP;
            {
                const uint32_t id_full = idesc_f16(128, 2 * NP), id_half = idesc_f16(128, NP);
                const uint64_t a0 = sdesc(smem_u32(base));
                constexpr uint64_t LO = PACK ? 64 / 16 : 16384 / 16, B0 = C::A_BYTES / 16;  // descriptor units of 16 bytes
                bool ok = true;
                for (int w = m, i = 0; ok && w < nv; w += NM, i++) {
                    const int gi = i + C::OFF * m, g = gi / C::GV, b = m * C::AC + g % C::AC;
                    const bool start = gi % C::GV == 0 || i == 0;
                    if (start && g >= C::AC) ok = mbar_wait_or(&acc_empty[b], (uint32_t)((g / C::AC - 1) & 1), abort_flag);
                    const uint32_t dmain = tmem + (uint32_t)(b * 2 * NP), dcorr = dmain + NP;
#pragma unroll
                    for (int kb = 0; kb < KB; kb++) {
                        const int u = w * KB + kb, s = u % NS;
                        const uint32_t ph = (uint32_t)((u / NS) & 1);
                        ok = ok && mbar_wait_or(&full[s], ph, abort_flag);
                        if (!lat) {
                            ok = ok && mbar_wait_or(&gfull[s], ph, abort_flag);
                            fence_proxy_async();  // the gathered rows (generic proxy) before the MMA's reads
                        }
                        ok = __all_sync(0xffffffffu, ok);
                        if (!ok) break;
                        tc_fence_after();
                        if (elect_one()) {
                            const uint64_t ad = a0 + (uint64_t)((uint32_t)s * (C::STAGE / 16)), bd = ad + B0;
                            const uint32_t first = (start && kb == 0) ? 0u : 1u;
                            // k-steps of 16 coefficients holding any of the p^2 real ones
                            constexpr int KS = PACK ? NP / 16 : 4;
                            const int ks = min(KS, (PP - kb * 64 + 15) >> 4);
#pragma unroll
                            for (int k = 0; k < KS; k++) {
                                if (k >= ks) break;
                                const uint32_t acc = k == 0 ? first : 1u;
                                // A_hi [T_hi ; T_lo] -> main | correction, then A_lo T_hi -> correction
                                if (PACK) {
                                    mma_f16(dmain, ad + 2 * k, bd + 2 * k, id_half, acc);
                                    mma_f16(dcorr, ad + 2 * k, bd + LO + 2 * k, id_half, acc);
                                } else {
                                    mma_f16(dmain, ad + 2 * k, bd + 2 * k, id_full, acc);
                                }
                                mma_f16(dcorr, ad + LO + 2 * k, bd + 2 * k, id_half, 1u);
                            }
                            mma_commit(&empty[s]);
                        }
                        __syncwarp();
                    }
                    if (ok && (gi % C::GV == C::GV - 1 || w + NM >= nv) && elect_one()) mma_commit(&acc_full[b]);
                    __syncwarp();
                }
                if (!ok) atomicExch(abort_flag, 1);
                // every commit has arrived before the shared memory goes away
                if (elect_one()) mma_commit(&fin[m]);
                mbar_wait(&fin[m], 0);
            }
            __syncwarp();
        } else {
            // ------------------------------------------------------ producer warps
            const int pw = warp - C::P_WARP;
            if (lane == 0 && pw < NM && nunits > pw) {
                int ox = 0, oy = 0, oz = 0;  // tile origin in halved coordinates
                const int obx = td.octant & 1, oby = (td.octant >> 1) & 1, obz = (td.octant >> 2) & 1;
                const unsigned char *lmap = nullptr;
                if (lat) {
                    // its first position, 128 td.block in Morton order
                    const unsigned k = (unsigned)td.block * C::M;
                    ox = (int)every_third(k);
                    oy = (int)every_third(k >> 1);
                    oz = (int)every_third(k >> 2);
                    lmap = J.lat_maps + 128 * l;
                }
                const unsigned char *ttab = J.ttab;
                int issued = pw;  // first unit of this producer not issued
                int4 vn = st[e0 + pw / KB];
                for (int u = pw; u < nunits; u += NM) {
                    const int s = u % NS, kb = u % KB;
                    const int4 v = vn;
                    if (u + NM < nunits) vn = st[e0 + (u + NM) / KB];
                    if (u >= NS && !mbar_wait_or(&empty[s], (uint32_t)((u / NS - 1) & 1), abort_flag)) {
                        atomicExch(abort_flag, 1);
                        break;
                    }
                    const uint32_t sa = smem_u32(base + s * C::STAGE);
                    mbar_arrive_tx(&full[s], C::B_BYTES + (lat ? C::A_BYTES : 0));
                    if (lat) {
                        // source octant bits and the block's shift in halved
                        // coordinates (arithmetic shifts: floor division by 2)
                        const int sx = obx + v.x, sy = oby + v.y, sz = obz + v.z;
                        const int ps = (sx & 1) | ((sy & 1) << 1) | ((sz & 1) << 2);
                        const int x = ox + (sx >> 1), y = oy + (sy >> 1), z = oz + (sz >> 1);
                        tma_load_5d(sa, lmap, kb * (C::ROWB / 2), x, y, z, ps, &full[s]);
                        if (!PACK) tma_load_5d(sa + 16384, lmap, kb * (C::ROWB / 2) + 64, x, y, z, ps, &full[s]);
                    }
                    bulk_g2s(sa + C::A_BYTES, ttab + ((size_t)(v.w & 0xffff) * KB + kb) * C::B_BYTES, C::B_BYTES, &full[s]);
                    issued = u + NM;
                }
                // copies still in flight when the pipeline stopped early land
                // before the shared memory goes away (bounded waits)
                if (*(volatile int *)abort_flag)
                    for (int u = pw; u < issued; u += NM)
                        if (u + NS >= issued) mbar_wait(&full[u % NS], (uint32_t)((u / NS) & 1));
            }
            __syncwarp();
        }
    } else {
        // ---------------------------------------------------------- worker warps
        if constexpr (!PERSIST && C::REGS) asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(C::REG_W));
        constexpr int HN = C::HN;
        const int row = tid & 127, g = (tid >> 7) & 1;  // target row and group
        float acc_hi[HN], acc_lo[HN];
#pragma unroll
        for (int k = 0; k < HN; k++) acc_hi[k] = acc_lo[k] = 0.f;
        const uint32_t tlane = (uint32_t)((warp & 3) * 32) << 16;  // this warp's TMEM lane quarter
        // this row's cell, its level, lattice position and octant (a pooled
        // tile mixes levels and octants)
        int px = 0, py = 0, pz = 0, cell = -1, rl = l, ro = 0;
        if (row < td.count) cell = J.tgt[td.start + row];  // (-1: a lattice position without a cell)
        if (cell >= 0) {
            const int4 a = J.xyz[cell];
            rl = a.w;
            const int sh = FMM_MAXLEVEL - rl;
            px = a.x >> sh;
            py = a.y >> sh;
            pz = a.z >> sh;
            ro = (px & 1) | ((py & 1) << 1) | ((pz & 1) << 2);
        }

        // Groups are drained in the order of their last vectors: (warp 1, 0),
        // (0, 0), (1, 1), (0, 1), ...; a group past its warp's last is skipped.
        const int nd = NM * ((nv + NM * C::GV - 1) / (NM * C::GV) + 1);  // bound of the sequence
        auto warp_of = [&](int d) { return NM - 1 - d % NM; };
        auto last_vector = [&](int d) { return NM * ((d / NM + 1) * C::GV - C::OFF * warp_of(d) - 1) + warp_of(d); };
        auto drain = [&](int d) {
            const int m = warp_of(d), gg = d / NM, b = m * C::AC + gg % C::AC;
            const int nm = (nv - m + NM - 1) / NM;  // vectors of warp m
            if (nm <= 0 || gg >= (nm + C::OFF * m + C::GV - 1) / C::GV) return;
            __syncwarp();
            const bool ok = __all_sync(0xffffffffu, mbar_wait_or(&acc_full[b], (uint32_t)((gg / C::AC) & 1), abort_flag));
            if (!ok) {
                atomicExch(abort_flag, 1);
                return;
            }
            tc_fence_after();
            const uint32_t taddr = tmem + tlane + (uint32_t)(b * 2 * NP + g * HN);
            // columns per read: 8 where the sums alone take most registers
            constexpr int CH = HN % 16 == 0 && HN <= 32 ? 16 : 8;
            float mv[CH], cv[CH];
#pragma unroll
            for (int k0 = 0; k0 < HN; k0 += CH) {
                if constexpr (CH == 16) {
                    tmem_ld16(taddr + k0, mv);
                    tmem_ld16(taddr + NP + k0, cv);
                } else {
                    tmem_ld8(taddr + k0, mv);
                    tmem_ld8(taddr + NP + k0, cv);
                }
#pragma unroll
                for (int k = 0; k < CH; k++) two_sum_acc(acc_hi[k0 + k], acc_lo[k0 + k], mv[k] + cv[k]);
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&acc_empty[b]);
        };

        int drained = 0;
        if (!lat) {
            const LevelDesc LD = J.ld[rl];
            const int *__restrict__ map_pool = J.map_pool;
            const unsigned char *__restrict__ mrow = J.mrow;
            const int nown = nunits > g ? (nunits - g + 1) / 2 : 0;  // units u = g, g + 2, ... of this group
            int *myring = ring + g * RINGU * C::M;
            const bool dense = LD.map_off >= 0;  // the level has a map: lookups arrive by cp.async
            const bool whole = rl <= 10 && LD.end - LD.start == (1 << (3 * rl));  // every lattice cell present
            const bool bricks = dense && !whole && LD.up > 0;  // a map in bricks: the ancestor's cell first, then the brick's entry
            const bool two = __any_sync(0xffffffffu, bricks);
            // source cell of this row for the group's unit j, looked up QU units
            // ahead into ring slot j % RINGU (cp.async of the lattice-map entry,
            // or a search of the level's keys); only this thread reads the slot.
            // Of a map in bricks `first` brings the ancestor's cell 2 QU units ahead.
            // The stencil entry of the next call is loaded one call ahead (calls
            // come in order), so its latency is hidden
            int4 st_next = make_int4(0, 0, 0, 0), st_first = make_int4(0, 0, 0, 0);
            int st_next_j = -1, st_first_j = -1;
            const unsigned side = 1u << rl;
            auto first = [&](int j) {
                if (!two || j >= nown) return;
                const int4 v = st_first_j == j ? st_first : st[e0 + (2 * j + g) / KB];
                if (j + 1 < nown) {
                    st_first = st[e0 + (2 * (j + 1) + g) / KB];
                    st_first_j = j + 1;
                }
                if (!bricks || cell < 0) return;
                int *const slot = myring + (j % RINGU) * C::M + row;
                const int x = px + v.x, y = py + v.y, z = pz + v.z;
                if (((v.w >> (16 + ro)) & 1) && (unsigned)x < side && (unsigned)y < side && (unsigned)z < side)
                    cp_async4(smem_u32(slot), map_pool + LD.top_off +
                                                  morton3_10((uint32_t)(x >> LD.up), (uint32_t)(y >> LD.up), (uint32_t)(z >> LD.up)));
                else
                    *slot = -1;
            };
            auto fetch = [&](int j) {
                if (j >= nown) return;
                const int4 v = st_next_j == j ? st_next : st[e0 + (2 * j + g) / KB];
                if (j + 1 < nown) {
                    st_next = st[e0 + (2 * (j + 1) + g) / KB];
                    st_next_j = j + 1;
                }
                int *const slot = myring + (j % RINGU) * C::M + row;
                int r = -1;
                if (cell >= 0) {
                    const int x = px + v.x, y = py + v.y, z = pz + v.z;
                    if (bricks) {
                        const int a = *slot;
                        const uint32_t m = (1u << LD.up) - 1u;
                        if (a >= 0)
                            cp_async4(smem_u32(slot), map_pool + LD.map_off + ((long long)(a - LD.top_start) << (3 * LD.up)) +
                                                          morton3_10((uint32_t)x & m, (uint32_t)y & m, (uint32_t)z & m));
                        return;
                    }
                    if (((v.w >> (16 + ro)) & 1) && (unsigned)x < side && (unsigned)y < side && (unsigned)z < side) {
                        // a complete level holds every lattice cell in Morton order:
                        // the index follows from the position
                        const uint32_t k = morton3_10((uint32_t)x, (uint32_t)y, (uint32_t)z);
                        if (whole) {
                            *slot = LD.start + (int)k;
                            return;
                        }
                        if (dense) {
                            cp_async4(smem_u32(slot), map_pool + LD.map_off + k);
                            return;
                        }
                        r = level_lookup(LD, map_pool, J.anchor, rl, x, y, z);
                    }
                }
                *slot = r;
            };
            for (int j = 0; j < 2 * QU; j++) first(j);
            cp_async_commit();
            cp_async_wait_all();
            for (int j = 0; j < QU; j++) fetch(j);
            cp_async_commit();
            cp_async_wait_all();
            for (int j = 0; j < nown; j++) {
                if (*(volatile int *)abort_flag) break;
                const int u = 2 * j + g, s = u % NS, kb = u % KB;
                // the groups before the vector this unit's stage waits for
                while (u >= NS && last_vector(drained) + C::LATE < (u - NS) / KB && !*(volatile int *)abort_flag) {
                    drain(drained);
                    drained++;
                }
                const bool ok = u < NS || mbar_wait_or(&empty[s], (uint32_t)((u / NS - 1) & 1), abort_flag);
                if (!__all_sync(0xffffffffu, ok)) {
                    atomicExch(abort_flag, 1);
                    break;
                }
                // slot j was fetched with the copies of unit j - QU: all but the
                // QU - 1 latest groups of copies are complete
                cp_async_wait<QU - 1>();
                const int src = myring[(j % RINGU) * C::M + row];
                // The warp fills its own 32 rows: in copy i, groups of CL lanes
                // take the CL 16-byte chunks of consecutive rows, so one warp
                // instruction reads whole rows; the source of each row comes from
                // the lane that looked it up
                constexpr int CL = C::ROWB / 16;  // 16 (hi 8 | lo 8), PACK: 8
                const uint32_t sa = smem_u32(base + s * C::STAGE);
                const int ch = lane % CL, sub = lane / CL, r0 = row - lane;  // r0: the warp's first row
                const uint32_t part = sa + (uint32_t)((ch >> 3) * 16384);
                const unsigned char *colp = mrow + kb * C::ROWB + ch * 16;
#pragma unroll
                for (int i = 0; i < CL; i++) {
                    const int rr = r0 + (32 / CL) * i + sub;
                    const int sc = __shfl_sync(0xffffffffu, src, (32 / CL) * i + sub);
                    cp_async16(part + (uint32_t)rr * 128u + ((((uint32_t)ch & 7u) ^ ((uint32_t)rr & 7u)) << 4),
                               colp + (size_t)(sc >= 0 ? sc : 0) * (KB * C::ROWB), sc >= 0 ? 16u : 0u);
                }
                fetch(j + QU);
                first(j + 2 * QU);
                cp_async_arrive_noinc(&gfull[s]);
                cp_async_commit();
            }
            cp_async_wait_all();
            __syncwarp();
        }
        while (drained < nd && !*(volatile int *)abort_flag) {
            drain(drained);
            drained++;
        }
        // once every worker warp is here the flag is final: either a wait has
        // failed, or the last drain saw the last MMA and nothing is waiting
        named_barrier_sync(1, C::NW * 32);
        if (!*(volatile int *)abort_flag) {
            const int e = cell >= 0 ? m2l_exponent(J.ws[rl]) : 0;
            float *Lc = J.L + (size_t)(cell >= 0 ? cell : 0) * PP;
            // back from the operands' powers of two
            auto put = [&](int k, float x) {
                const int t = J.rowexp[k] - e;
                if (cell >= 0) Lc[k] += (x * m2l_pow2(t >> 1)) * m2l_pow2(t - (t >> 1));
            };
            if (nsplit == 1) {
#pragma unroll
                for (int k = 0; k < HN; k++)
                    if (g * HN + k < PP) put(g * HN + k, acc_hi[k] + acc_lo[k]);
            } else {
                // the range's sums, [item][coefficient][row]; the tile's last
                // range to finish adds them all in order
                const size_t rng = (size_t)PP * C::M;
                float2 *pt = J.part + (size_t)item * rng + row;
#pragma unroll
                for (int k = 0; k < HN; k++)
                    if (g * HN + k < PP) __stcg(&pt[(size_t)(g * HN + k) * C::M], make_float2(acc_hi[k], acc_lo[k]));
                __threadfence();
                named_barrier_sync(1, C::NW * 32);
                if (tid == 0) {
                    const bool last = atomicAdd(&J.tcnt[tile], 1u) == (unsigned)(nsplit - 1);
                    if (last) J.tcnt[tile] = 0u;
                    *s_last = last;
                    __threadfence();
                }
                named_barrier_sync(1, C::NW * 32);
                if (*(volatile int *)s_last) {
                    constexpr int CH = HN % 16 == 0 && HN <= 32 ? 16 : 8;  // coefficients in flight per range
                    const float2 *p0 = J.part + (size_t)tile * nsplit * rng + row;
                    for (int k0 = g * HN; k0 < (g + 1) * HN && k0 < PP; k0 += CH) {
                        float hi[CH], lo[CH];
#pragma unroll
                        for (int k = 0; k < CH; k++) hi[k] = lo[k] = 0.f;
#pragma unroll 2
                        for (int r = 0; r < nsplit; r++) {
                            float2 v[CH];
#pragma unroll
                            for (int k = 0; k < CH; k++)
                                v[k] = k0 + k < PP ? __ldcg(&p0[(size_t)r * rng + (size_t)(k0 + k) * C::M]) : make_float2(0.f, 0.f);
#pragma unroll
                            for (int k = 0; k < CH; k++) {
                                two_sum_acc(hi[k], lo[k], v[k].x);
                                lo[k] += v[k].y;
                            }
                        }
#pragma unroll
                        for (int k = 0; k < CH; k++)
                            if (k0 + k < PP) put(k0 + k, hi[k] + lo[k]);
                    }
                }
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const bool aborted = *(volatile int *)abort_flag != 0;
    if (tid == 0 && aborted) atomicExch(err, 1);
    __syncthreads();  // every thread has read the flag before the next item resets it
    if (aborted) break;
    }  // items
    tc_fence_before();
    __syncthreads();
    if (warp == C::MMA_WARP) {
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(C::TCOLS));
    }
    // the wide tiles of many systems, in turn over the CTAs
    if (PERSIST && *s_wide)
        for (int it = blockIdx.x; it < jobs[njobs - 1].item0 + jobs[njobs - 1].count; it += (int)gridDim.x) {
            const M2LJob &J = jobs[job_of(jobs, njobs, it)];
            if (m2l_is_wide(J.ws[M2LW_WIDE], J.tiles[(it - J.item0) / J.nsplit]))
                m2l_wide_tile<NP>(J, p, it - J.item0, *reinterpret_cast<WideShared<NP> *>(base));
        }
}

// ---------------------------------------------------------------------------
// host
// ---------------------------------------------------------------------------
// p^2 padded to the MMA's N; 0: not supported
static int tc_np(int p)
{
    const int PP = p * p;
    for (int np : {16, 32, 48, 64, 96, 112, 128})
        if (PP <= np) return np;
    return 0;
}
static int tc_kb(int p) { return (tc_np(p) + 63) / 64; }                      // k-blocks of 64 coefficients
static size_t tc_row_bytes(int p) { return (size_t)tc_kb(p) * (tc_np(p) <= 32 ? 128 : 256); }
static size_t tc_op_bytes(int p) { return (size_t)tc_kb(p) * (tc_np(p) <= 32 ? 1 : 2) * tc_np(p) * 128; }

bool tensor_m2l_supported(fmm_ctx *h) { return h->p >= 2 && tc_np(h->p) > 0 && h->cc_major == 10; }

// I_n^m(x) in full storage (n*n + n + m), degrees < Q, from the Cartesian
// recurrences of the irregular solid harmonics
static void build_irregular_full(int Q, double x, double y, double z, std::vector<double> &re, std::vector<double> &im)
{
    re.assign((size_t)Q * Q, 0.0);
    im.assign((size_t)Q * Q, 0.0);
    const double r2 = x * x + y * y + z * z, ir2 = 1.0 / r2;
    auto put = [&](int n, int m, double a, double b) {
        re[n * n + n + m] = a;
        im[n * n + n + m] = b;
        if (m) {
            const double sg = (m & 1) ? -1.0 : 1.0;
            re[n * n + n - m] = sg * a;
            im[n * n + n - m] = -sg * b;
        }
    };
    double mr = std::sqrt(ir2), mi = 0.0;
    for (int m = 0; m < Q; m++) {
        if (m > 0) {
            const double f = (double)(2 * m - 1) * ir2;
            const double a = (mr * x - mi * y) * f, b = (mr * y + mi * x) * f;
            mr = a;
            mi = b;
        }
        put(m, m, mr, mi);
        if (m + 1 >= Q) continue;
        const double f1 = (double)(2 * m + 1) * z * ir2;
        double p2r = mr, p2i = mi, p1r = mr * f1, p1i = mi * f1;
        put(m + 1, m, p1r, p1i);
        for (int n = m + 2; n < Q; n++) {
            const double a = (double)(2 * n - 1) * z, b = (double)((n + m - 1) * (n - m - 1));
            const double cr = (a * p1r - b * p2r) * ir2, ci = (a * p1i - b * p2i) * ir2;
            put(n, m, cr, ci);
            p2r = p1r;
            p2i = p1i;
            p1r = cr;
            p1i = ci;
        }
    }
}

// The operators of every stencil vector: the real p^2 x p^2 map of M2L in the
// packed layout, L~_n^m = (-1)^n sum_{j,k} M~_j^k I_{j+n}^{k+m}(u), u = -v,
// its columns divided by m2l_norm and its rows multiplied by 2^-rowexp (a
// factorial part as for the columns, and a part per degree that brings the
// largest entries of the degree into [2^13, 2^14)), then split into FP16 (hi,
// lo) and laid out as the 128B-swizzled shared-memory image of the B operand:
// per k-block of 64 columns, rows 0..NP-1 = T_hi, rows NP..2NP-1 = T_lo (NP <=
// 32: rows of T_hi | T_lo). The rowexp of the coefficients follow the vectors.
// It depends only on p and the stencil, which the MAC constant and the
// stencil bound fix (vectors are numbered in a fixed order): the host image is
// built once per process, and the handles of one device that use it share one
// device copy, which lives as long as the last of them (a batch's tiles then
// find the operators of every system in L2).
struct TcImage {
    DevBuf buf;
    ~TcImage() { buf.release(); }
};
using HostImage = std::vector<unsigned char>;

static std::mutex g_img_mu;
static std::map<std::tuple<int, double, int>, std::shared_ptr<const HostImage>> g_img_cache;
static std::map<std::tuple<int, double, int, int>, std::weak_ptr<TcImage>> g_dev_img;

static std::shared_ptr<const HostImage> build_image(fmm_ctx *h)
{
    const int p = h->p, PP = p * p, Q = 2 * p - 1, NP = tc_np(p);
    const bool pack = NP <= 32;
    const size_t per_v = tc_op_bytes(p), bbytes = per_v / tc_kb(p);
    auto img = std::make_shared<HostImage>();
    img->assign((size_t)h->nV * per_v + sizeof(int) * M2L_NORM_N, 0);
    std::vector<int> seen(h->nV, 0);
    std::vector<double> Ire, Iim, T((size_t)PP * PP);
    auto re_i = [](int n, int m) { return n * n + (m == 0 ? 0 : 2 * m - 1); };
    auto im_i = [](int n, int m) { return n * n + 2 * m; };
    const int ne = h->st_off[8];
    auto make = [&](int vx, int vy, int vz) {
        build_irregular_full(Q, -(double)vx, -(double)vy, -(double)vz, Ire, Iim);
        auto I = [&](int n, int m, double &r, double &i) {
            r = Ire[n * n + n + m];
            i = Iim[n * n + n + m];
        };
        std::fill(T.begin(), T.end(), 0.0);
        for (int j = 0; j < p; j++)
            for (int k = 0; k <= j; k++)
                for (int part = 0; part < (k ? 2 : 1); part++) {
                    // M_j^k = e (1 or i), M_j^{-k} = (-1)^k conj(e)
                    const double er = part ? 0.0 : 1.0, ei = part ? 1.0 : 0.0;
                    const int col = part ? im_i(j, k) : re_i(j, k);
                    for (int n = 0; n < p; n++)
                        for (int m = 0; m <= n; m++) {
                            double ir, ii, sr, si;
                            I(j + n, k + m, ir, ii);
                            sr = er * ir - ei * ii;
                            si = er * ii + ei * ir;
                            if (k) {
                                const double sg = (k & 1) ? -1.0 : 1.0;
                                double jr, ji;
                                I(j + n, m - k, jr, ji);
                                const double cr = sg * er, ci = -sg * ei;  // (-1)^k conj(e)
                                sr += cr * jr - ci * ji;
                                si += cr * ji + ci * jr;
                            }
                            if (n & 1) {
                                sr = -sr;
                                si = -si;
                            }
                            T[(size_t)re_i(n, m) * PP + col] = sr;
                            if (m) T[(size_t)im_i(n, m) * PP + col] = si;
                        }
                }
        for (int r = 0; r < PP; r++)
            for (int c = 0; c < PP; c++)
                T[(size_t)r * PP + c] = std::ldexp(T[(size_t)r * PP + c], -(m2l_fact_exp(r) + m2l_norm_exp(c)));
    };
    // the entries decay with the distance: a degree's largest belongs to the
    // shortest vectors (with the factor of 4 that [2^13, 2^14) leaves to FP16's
    // largest value, beyond which the build of the image would fail)
    double d2min = 1e300, big[FMM_MAXP] = {};
    auto d2 = [&](int e) {
        const int *v = &h->st_host[4 * (size_t)e];
        return (double)v[0] * v[0] + (double)v[1] * v[1] + (double)v[2] * v[2];
    };
    for (int e = 0; e < ne; e++) d2min = std::min(d2min, d2(e));
    for (int e = 0; e < ne; e++) {
        const int *v = &h->st_host[4 * (size_t)e];
        if (seen[v[3] & 0xffff] || d2(e) > 2.0 * d2min) continue;
        seen[v[3] & 0xffff] = 1;
        make(v[0], v[1], v[2]);
        for (int n = 0; n < p; n++)
            for (size_t i = (size_t)n * n * PP; i < (size_t)(n + 1) * (n + 1) * PP; i++) big[n] = std::max(big[n], std::fabs(T[i]));
    }
    std::fill(seen.begin(), seen.end(), 0);
    std::vector<int> rexp(M2L_NORM_N, 0), rowexp(M2L_NORM_N, 0);
    for (int n = 0; n < p; n++)
        for (int r = n * n; r < (n + 1) * (n + 1); r++) {
            rexp[r] = big[n] > 0 ? 13 - std::ilogb(big[n]) : 0;
            rowexp[r] = m2l_fact_exp(r) - rexp[r];
        }
    memcpy(img->data() + (size_t)h->nV * per_v, rowexp.data(), sizeof(int) * M2L_NORM_N);
    for (int e = 0; e < ne; e++) {
        const int *v = &h->st_host[4 * (size_t)e];
        const int id = v[3] & 0xffff;
        if (seen[id]) continue;
        seen[id] = 1;
        make(v[0], v[1], v[2]);
        unsigned char *dst = img->data() + (size_t)id * per_v;
        for (int r = 0; r < PP; r++)
            for (int c = 0; c < PP; c++) {
                const double t = std::ldexp(T[(size_t)r * PP + c], rexp[r]);
                if (!(std::fabs(t) < 65504.0)) throw Error{FMM_EINVAL, "tensor-core M2L: operator entry beyond FP16"};
                const __half hi = __float2half_rn((float)t);
                const __half lo = __float2half_rn((float)(t - (double)__half2float(hi)));
                const int kb = pack ? 0 : c >> 6;
                for (int part = 0; part < 2; part++) {
                    const int row = pack ? r : r + part * NP, cc = pack ? c + 32 * part : c & 63;
                    const size_t off = (size_t)kb * bbytes + (size_t)row * 128 + (size_t)((((cc >> 3) ^ (row & 7)) << 4) + (cc & 7) * 2);
                    const __half x = part ? lo : hi;
                    memcpy(dst + off, &x, 2);
                }
            }
    }
    return img;
}

void tensor_tables_update(fmm_ctx *h)
{
    if (!tc_np(h->p)) return;
    if (h->ttab_nv == h->nV && h->ttab) return;
    std::lock_guard<std::mutex> lk(g_img_mu);
    auto &dev = g_dev_img[std::make_tuple(h->p, h->cmac, h->st_R, h->dev)];
    std::shared_ptr<TcImage> img = dev.lock();
    if (!img) {
        auto &host = g_img_cache[std::make_tuple(h->p, h->cmac, h->st_R)];
        if (!host) host = build_image(h);
        img = std::make_shared<TcImage>();
        img->buf.ensure(host->size());
        FMM_CUDA_TRY(cudaMemcpy(img->buf.p, host->data(), host->size(), cudaMemcpyHostToDevice));
        // handles on other streams may read the copy as soon as it is shared
        FMM_CUDA_TRY(cudaStreamSynchronize(cudaStreamLegacy));
        dev = img;
    }
    h->ttab = img;
    h->ttab_nv = h->nV;
}

template <int NP>
static void launch_tc(int p, int grid, const M2LJob &one, const M2LJob *jobs, int njobs, int *queue, const unsigned *any,
                      int *err, cudaStream_t s)
{
    using C = TcCfg<NP>;
    // grid: one CTA per SM with a job list (persistent), else one per item
    if (jobs) {
        ensure_smem((const void *)m2l_tc_k<NP, true>, C::SMEM);
        FMM_CUDA_TRY(cudaMemsetAsync(queue, 0, sizeof(int), s));
        m2l_tc_k<NP, true><<<grid, C::NT, C::SMEM, s>>>(p, one, jobs, njobs, queue, any, err);
    } else {
        ensure_smem((const void *)m2l_tc_k<NP, false>, C::SMEM);
        // the workers' registers come out of the launch's: with fewer they would wait for ever
        static const bool fits = [] {
            cudaFuncAttributes a;
            return cudaFuncGetAttributes(&a, (const void *)m2l_tc_k<NP, false>) == cudaSuccess &&
                   a.numRegs * C::NT >= 32 * (C::NW * C::REG_W + 4 * C::REG_O);
        }();
        if (C::REGS && !fits) throw Error{FMM_ECUDA, "tensor-core M2L: too few registers at launch"};
        m2l_tc_k<NP, false><<<grid, C::NT, C::SMEM, s>>>(p, one, jobs, njobs, queue, any, err);
    }
}

#define FMM_TC_SWITCH(np, CALL)                                            \
    switch (np) {                                                          \
    case 16: CALL(16); break;                                              \
    case 32: CALL(32); break;                                              \
    case 48: CALL(48); break;                                              \
    case 64: CALL(64); break;                                              \
    case 96: CALL(96); break;                                              \
    case 112: CALL(112); break;                                            \
    case 128: CALL(128); break;                                            \
    default: throw Error{FMM_EINVAL, "tensor-core M2L: unsupported p"};    \
    }

static void launch_tc_p(int p, int grid, const M2LJob &one, const M2LJob *jobs, int njobs, int *queue, const unsigned *any,
                        int *err, cudaStream_t s)
{
#define FMM_TC_CALL(NPV) launch_tc<NPV>(p, grid, one, jobs, njobs, queue, any, err, s)
    FMM_TC_SWITCH(tc_np(p), FMM_TC_CALL)
#undef FMM_TC_CALL
}

// the longest list of vectors that a tile of the tree walks
int m2l_longest_list(fmm_ctx *h)
{
    const int pool_max = h->m2l_pool >= 0 ? h->m2l_pool : 4 * m2l_tile_size(h);
    int nv = 1;
    for (int l = 2; l <= h->depth; l++) {
        const bool pooled = h->lvl_start[(size_t)l + 1] - h->lvl_start[(size_t)l] <= pool_max;
        for (int o = pooled ? 8 : 0; o < (pooled ? 9 : 8); o++)
            nv = std::max(nv, h->st_cnt[(size_t)o * (FMM_MAXLEVEL + 1) + l]);
    }
    return nv;
}

// How many ranges the vectors of every tile are cut into. A CTA's time is
// about (its vectors + 10) units, one unit a vector's copies (+ 13 with its
// sums' way through memory), plus one per range for the last CTA's sum of them; the launch takes the waves of
// ntiles x nsplit CTAs over the SMs. One range wins as soon as the tiles fill
// a few waves. Ranges are whole drain groups of both MMA warps.
void m2l_plan(fmm_ctx *h)
{
    h->m2l_nsplit = 1;
    h->m2l_chunk = INT_MAX;
    if (h->precision != FMM_MIXED || h->engine_used != FMM_M2L_TENSOR || h->ntiles_max < 1) return;
    const int nv = m2l_longest_list(h);
    double best = 1e300;
    for (int want = 1; want <= 32; want++) {
        constexpr int G = 2 * TcCfg<64>::GV;
        const int chunk = (nv + want * G - 1) / (want * G) * G, s = (nv + chunk - 1) / chunk;
        const double waves = (double)(((int64_t)h->m2l_plan_tiles * s + h->nsm - 1) / h->nsm);
        const double t = waves * ((double)std::min(chunk, nv) + (s > 1 ? 13.0 : 10.0)) + (s > 1 ? s : 0);
        if (t < best) {
            best = t;
            h->m2l_nsplit = s;
            h->m2l_chunk = chunk;
        }
    }
}

M2LJob m2l_tensor_job(fmm_ctx *h, float *L)
{
    tensor_tables_update(h);
    const int nc = h->ncells;
    h->msplit.ensure(tc_row_bytes(h->p) * (size_t)nc);
    h->m2l_ws.ensure(sizeof(unsigned) * (M2LW_CNT + (size_t)h->ntiles_max + (size_t)nc));
    if (h->m2l_nsplit > 1)
        h->m2l_part.ensure(sizeof(float2) * (size_t)h->ntiles_max * h->m2l_nsplit * h->p * h->p * TcCfg<64>::M);
    M2LJob j;
    j.tiles = h->m2l_tiles.as<M2LTile>();
    j.ntiles = reinterpret_cast<const int *>(h->m2l_misc.as<unsigned>() + 24 * (FMM_MAXLEVEL + 1));
    j.tgt = h->m2l_tgt.as<int>();
    j.xyz = h->c_xyz.as<int4>();
    j.anchor = h->c_anchor.as<uint64_t>();
    j.ld = h->lvl_desc.as<LevelDesc>();
    j.map_pool = h->map_pool.as<int>();
    j.st = h->st_dev.as<int4>();
    j.st_off = stencil_offsets(h);
    j.mrow = h->msplit.as<unsigned char>();
    j.ttab = h->ttab->buf.as<unsigned char>();
    j.L = L;
    j.M = h->Mexp.as<float>();
    j.ws = h->m2l_ws.as<unsigned>();
    j.tcnt = h->m2l_ws.as<unsigned>() + M2LW_CNT;
    j.ws_words = M2LW_CNT + h->ntiles_max;
    j.cmax = h->m2l_ws.as<unsigned>() + j.ws_words;
    j.part = h->m2l_part.as<float2>();
    j.nsplit = h->m2l_nsplit;
    j.chunk = h->m2l_chunk;
    j.rowexp = reinterpret_cast<const int *>(j.ttab + (size_t)h->nV * tc_op_bytes(h->p));
    j.lat_maps = nullptr;  // gathers on every level (the single-system launch sets the lattice maps)
    j.item0 = 0;
    j.count = -1;
    return j;
}

// cuTensorMapEncodeTiled, looked up once through the runtime (no link
// against the driver library)
using EncodeTiledFn = CUresult (*)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                   const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                   CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

static EncodeTiledFn encode_tiled()
{
    static EncodeTiledFn fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void *f = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(f);
    });
    return fn;
}

// Lattice levels: at least three quarters of the positions hold a cell, at
// least 8^4 positions, more cells than the pooling threshold, level 9 at most.
// Their tiles are blocks of 128 positions of one octant, with or without a
// cell, and read their sources by TMA from the lattice copy of the level's
// rows, zeros where there is no cell. A tile by TMA takes about 0.45 of the
// time of one with gathered rows (N = 1e6 Plummer against uniform trees), so
// the rows without a cell should cost less than the gathers from half full on;
// the line lies higher because the batch engine, which gathers on every level,
// pays for them (a third more rows at most). M2L at N = 3e5
// uniform, p = 8, whose level 5 is 85 % full: 2.66 -> 2.14 ms.
static unsigned dense_levels(fmm_ctx *h, int pool_max)
{
    unsigned m = 0;
    for (int l = 4; l <= std::min(h->depth, 9); l++) {
        const long long cells = (long long)h->lvl_start[(size_t)l + 1] - h->lvl_start[(size_t)l];
        if (4 * cells >= 3ll << (3 * l) && cells > pool_max) m |= 1u << l;
    }
    return m;
}

// tiles of the tree with every such level in lattice tiles
static int plan_tiles(fmm_ctx *h)
{
    constexpr int M = TcCfg<64>::M;
    const int pool_max = h->m2l_pool >= 0 ? h->m2l_pool : 4 * M;
    const unsigned dense = dense_levels(h, pool_max);
    int64_t pooled = 0, nt = 0;
    for (int l = 2; l <= h->depth; l++) {
        const int cells = h->lvl_start[(size_t)l + 1] - h->lvl_start[(size_t)l];
        if (cells <= pool_max) pooled += cells;
        else nt += (dense >> l) & 1u ? (1ll << (3 * l)) / M : cells / M + 8;
    }
    return (int)(nt + (pooled + M - 1) / M);
}

void lattice_select(fmm_ctx *h, int pool_max)
{
    h->lat_levels = h->lat_complete = 0;
    // the ranges of the vectors are planned for these tiles with or without the
    // lattice loads, whose results are then the same bit for bit
    const unsigned dense = dense_levels(h, pool_max);
    h->m2l_plan_tiles = plan_tiles(h);
    if (!h->lattice_req || h->precision != FMM_MIXED || h->engine_used != FMM_M2L_TENSOR || !tensor_m2l_supported(h) ||
        m2l_tile_size(h) != TcCfg<64>::M || !encode_tiled())
        return;
    long long total = 0;
    for (int l = 4; l <= std::min(h->depth, 9); l++) {
        const long long cells = (long long)h->lvl_start[(size_t)l + 1] - h->lvl_start[(size_t)l], all = 1ll << (3 * l);
        if (!((dense >> l) & 1u)) continue;
        h->lat_levels |= 1u << l;
        if (cells == all) h->lat_complete |= 1u << l;
        h->lat_off[l] = total;
        total += all;
    }
    h->lat_rows = total;
}

// One 5-D tensor map per lattice level over [octant bits][z/2][y/2][x/2][row]
// (FP16), box 64 halves x 8 x 4 x 4 x 1 = one half (hi or lo) of the tile's 128
// rows, 128-byte swizzle (the layout of the gathered stages).
void lattice_prepare(fmm_ctx *h, cudaStream_t s)
{
    const unsigned levels = h->lat_levels;
    if (!levels) return;
    const EncodeTiledFn enc = encode_tiled();
    const cuuint64_t row = tc_row_bytes(h->p);
    const long long total = h->lat_rows;
    h->mlat.ensure((size_t)row * (size_t)total);
    // rows of positions without a cell, which no evaluation writes
    for (int l = 4; l <= 9; l++)
        if (((levels & ~h->lat_complete) >> l) & 1u)
            FMM_CUDA_TRY(cudaMemsetAsync(h->mlat.as<unsigned char>() + row * h->lat_off[l], 0, (size_t)row << (3 * l), s));
    const size_t mbytes = sizeof(CUtensorMap) * (FMM_MAXLEVEL + 1);
    h->lat_maps.ensure(mbytes);
    h->lat_host.ensure(mbytes);
    CUtensorMap *mp = h->lat_host.as<CUtensorMap>();
    std::memset(mp, 0, mbytes);
    for (int l = 4; l <= 9; l++) {
        if (!((levels >> l) & 1u)) continue;
        const cuuint64_t H = 1ull << (l - 1);
        const cuuint64_t dims[5] = {row / 2, H, H, H, 8};
        const cuuint64_t strides[4] = {row, row * H, row * H * H, row * H * H * H};
        const cuuint32_t box[5] = {64, 8, 4, 4, 1}, estride[5] = {1, 1, 1, 1, 1};
        const CUresult r = enc(&mp[l], CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 5, h->mlat.as<unsigned char>() + row * h->lat_off[l],
                               dims, strides, box, estride, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                               CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
        if (r != CUDA_SUCCESS) throw Error{FMM_ECUDA, "tensor-core M2L: encoding a lattice tensor map failed"};
    }
    FMM_CUDA_TRY(cudaMemcpyAsync(h->lat_maps.p, mp, mbytes, cudaMemcpyHostToDevice, s));
}

template <int NP>
__global__ void __launch_bounds__(256) batch_split_k(int PP, const BatchSys *__restrict__ sys, unsigned *any)
{
    using C = TcCfg<NP>;
    constexpr int NCH = NP / 8;
    const BatchSys &S = sys[blockIdx.y];
    if (!S.rows || S.c0 >= S.ncells) return;
    const int64_t cnt = (int64_t)(S.ncells - S.c0) * NCH;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < cnt; i += (int64_t)gridDim.x * blockDim.x) {
        const int c = S.c0 + (int)(i / NCH), ch = (int)(i % NCH), l = S.xyz[c].w;
        m2l_split_chunk<NP>(S.M + (size_t)c * PP, PP, ch, m2l_exponent(S.m2l_ws[l]), S.rows + (size_t)c * (C::KB * C::ROWB));
        if (ch == 0) m2l_mark(c, l, S.m2l_cmax, S.parent, S.m2l_ws, any);
    }
}

void batch_split(int p, const BatchSys *sys, int nsys, unsigned *any, cudaStream_t s)
{
#define FMM_TC_CALL(NPV) batch_split_k<NPV><<<dim3(16, (unsigned)nsys), 256, 0, s>>>(p *p, sys, any)
    FMM_TC_SWITCH(tc_np(p), FMM_TC_CALL)
#undef FMM_TC_CALL
    check_launch("batch split");
}

void m2l_tensor_jobs(int p, int nsm, const M2LJob *jobs_dev, int njobs, int *queue, const unsigned *any, int *err,
                     cudaStream_t s)
{
    M2LJob none;
    std::memset(&none, 0, sizeof(none));
    launch_tc_p(p, nsm, none, jobs_dev, njobs, queue, any, err, s);
}

void m2l_tensor(fmm_ctx *h, float *L, const float *M)
{
    cudaStream_t s = h->work;
    M2LJob j = m2l_tensor_job(h, L);
    const int PP = h->p * h->p, nc = h->ncells, c0 = h->lvl_start[2];
    int *misc = reinterpret_cast<int *>(h->m2l_misc.as<unsigned>() + 24 * (FMM_MAXLEVEL + 1));
    int *err = misc + 4, *queue = misc + 6;
    FMM_CUDA_TRY(cudaMemsetAsync(err, 0, sizeof(int), s));
    if (nc <= c0) return;
    FMM_CUDA_TRY(cudaMemsetAsync(h->m2l_ws.p, 0, sizeof(unsigned) * (size_t)j.ws_words, s));
    M2LLevels lv;
    int most = 0;
    for (int l = 0; l <= FMM_MAXLEVEL + 1; l++) {
        lv.start[l] = l < (int)h->lvl_start.size() ? h->lvl_start[(size_t)l] : nc;
        if (l) most = std::max(most, lv.start[l] - lv.start[l - 1]);
    }
    // a block walks 64 cells or more; 4 blocks per SM at most
    const unsigned gx = (unsigned)std::min((most + 63) / 64, 4 * h->nsm);
    m2l_lmax_k<<<dim3(gx, (unsigned)h->depth - 1), 256, 0, s>>>(M, PP, lv, const_cast<unsigned *>(j.cmax), h->m2l_ws.as<unsigned>());
    count_launch(h);
    M2LLattice lat;
    lat.levels = h->lat_levels;
    for (int l = 0; l <= FMM_MAXLEVEL; l++) lat.off[l] = h->lat_off[l];
#define FMM_TC_CALL(NPV)                                                                                           \
    m2l_split_k<NPV><<<nblk((int64_t)(nc - c0) * (NPV / 8), 256), 256, 0, s>>>(                                     \
        M, PP, h->c_xyz.as<int4>(), c0, nc, h->c_parent.as<int>(), j.cmax,                                           \
        h->m2l_ws.as<unsigned>(), lat, h->msplit.as<unsigned char>(), h->mlat.as<unsigned char>())
    FMM_TC_SWITCH(tc_np(h->p), FMM_TC_CALL)
#undef FMM_TC_CALL
    count_launch(h);
    if (h->lat_levels) {
        j.lat_maps = h->lat_maps.as<unsigned char>();
    }
    launch_tc_p(h->p, h->ntiles_max * j.nsplit, j, nullptr, 1, queue, j.ws + M2LW_WIDE, err, s);
    count_launch(h);
    check_launch("m2l tensor");
}

}  // namespace fmm
