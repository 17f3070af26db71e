// The Kronecker-product transforms of the mixed-precision inner Poisson
// solve on the fifth-generation tensor cores (tcgen05).
//
// Sec. II.A writes the finite-difference Laplacian as a Kronecker sum; its
// inverse is three forward 1-D transforms, a diagonal scaling and three
// inverse transforms (kron.cu has the algebra and the CUDA-core kernel).
// Each transform multiplies every line of one direction by a dense matrix:
// a GEMM with K = the line length, so it belongs on the tensor cores.
//
// Layout.  A pass reads its input as rows (one row = one line, its n points
// contiguous) and writes its output transposed: out[orb][k][row], k the
// position (or mode) along the line.  The three directions therefore rotate
// through the passes: the standard [z][y][x] input r becomes [mx][z][y]
// after the x pass, [my][mx][z] after the y pass, [mz][my][mx] after the z
// pass (with the scaling), [x][mz][my], [y][x][mz] and finally the standard
// [z][y][x] after the inverse x, y and z passes.  Every side n is padded to
// p (kron_pad: a multiple of 4, p = n when n is a multiple of 8), in every
// layout, so that each row starts on a 16-byte boundary and any side will
// do: the even modes of a line sit at [0, ns), the odd ones at [ns4, ns4 +
// na) with ns4 = ns rounded up to 4.  The padding is never
// initialised and may hold anything, NaN too: a row only ever reaches its own
// results (padding rows end in padding rows), and the padding elements of a line
// are dropped by selection, not by a product, when the line is read and when
// results are stored.  Every input row is a contiguous run that one tiled bulk copy
// (TMA, 128-byte swizzle) brings to shared memory; every output store is
// coalesced (the 32 lanes of a warp own 32 consecutive rows).
//
// One CTA per SM (14 warps) streams tiles of 128 rows.  The copy engine
// delivers a tile's rows (float32) into a ring of 32-point boxes, up to two
// tiles ahead.  Eight converter warps fold each row into its even and odd
// halves (s_k = v_k + v_{n-1-k}, a_k = v_k - v_{n-1-k}: T_d commutes with the
// reflection, so the transform splits into two half-size products) and write
// each half as three bf16 terms (v = v1 + v2 + v3, ~24 significant bits)
// straight into tensor memory, the MMAs' A operand (row i in lane i); the
// split matrices stay in shared memory (B operand, K-major).  One warp issues
// the copies, another the MMAs: per unit of 32 modes of one half, the six
// split products v_i w_j with i + j <= 2, the v1 w1 product into its own
// accumulator and the five smaller ones into a second.  Units rotate through
// a ring of accumulators, so the MMAs run ahead while the four epilogue
// warps read a pair of units back (tcgen05.ld), apply the scaling (forward z)
// or the even/odd recombination (inverse) and store (128 bytes per line and
// warp; staging the lines for bulk stores cost more in fences than it saved).
//
// Two instances: half-lines of up to 64 points (sides <= 128: two tiles of
// staged rows, four units in flight) and of up to 96 (sides <= 192: one
// tile, three units; the matrices take 108 KB).
//
// What bounds it: 8 B per point and pass, a 128-row tile of 128-point lines
// 5.6k cycles of an SM's share of HBM; the roles run concurrently, each about
// 4 to 6k cycles per tile (converting 4k, MMA issue 3k, epilogue 5k of which
// 2k are the stores' own rate).  At 128^3 x 64 a solve's 6.4 GB take 1.31 ms
// (0.72 of the measured copy rate; 1.77 with the MMAs issued from a lane-0
// branch, one accumulator per half and staged bulk stores).  Against the
// CUDA-core kernel: 192^3 x 24 7.35 -> 1.82 ms per solve, 117^3 x 20 1.35 ->
// 0.44 ms.
//
// Accuracy: keeping the dominant product in its own short accumulation
// chain (one instruction of K = 16 per 16 points of a half) holds the tensor
// cores' float32 accumulation error to the level of a float32 CUDA-core
// product, so two refinement rounds still reach 1e-10.
//
// Which blocks: see kron_tc_eligible.  Every mbarrier wait is bounded; a
// timeout sets bit 4 of status word 3, lets the CTA wait (bounded) for its
// copies and MMAs in flight, frees its tensor memory and return.
#include <cuda_bf16.h>

#include <cmath>
#include <cstring>
#include <vector>

#include "internal.cuh"
#include "tcgen05.cuh"

namespace flosic {
namespace {

constexpr int kTcRows = 128;                      // rows (lines) per tile: MMA M
constexpr int kTcUnit = 32;                       // modes per accumulator unit: MMA N
constexpr int kTcConv = 256;                      // converter threads (warps 1-8: two per row)
constexpr int kTcThreads = 32 + kTcConv + 128 + 32;   // MMA warp, converters, epilogue (warps 9-12), copy warp
constexpr int kTcBox = kTcRows * 32 * 4;          // one copy: 128 rows x 32 points (float32): 16 KB
constexpr int kTcInfo = 16;                       // ring of tile descriptors
constexpr uint32_t kTcCols = 512;                 // tensor-memory columns

// Shapes of the instance for half-lines of up to HP points.
template <int HP>
struct TcShape {
    static constexpr int kKC = HP <= 64 ? 0 : HP - 64;          // K beyond the first 64 (64-byte swizzled rows)
    static constexpr int kBTile = HP * 128 + HP * 2 * kKC;      // one split of one half-matrix (bf16)
    static constexpr int kBoxes = HP <= 64 ? 9 : 7;             // staged boxes (ring)
    static constexpr int kUnits = HP <= 64 ? 4 : 3;             // accumulator units (ring)
    static constexpr int kOffRaw = 6 * kBTile;
    static constexpr int kSmem = kOffRaw + kBoxes * kTcBox + 1024;   // + alignment slack
    static constexpr uint32_t kColA = kUnits * 2 * kTcUnit;     // A operands: half h, split s at + (HP / 2)(3 h + s)
    static constexpr int kMatElems = HP * HP;                   // one padded half-matrix
    static constexpr int kPre = HP <= 64 ? 4 : 3;               // groups of 8 K values a converter folds ahead
    // HP 64: a tile's units are issued half by half, so a half is converted while
    // the other one's MMAs run (two chunks: four units hold a tile).  HP 96: chunk by
    // chunk (three units), after both halves have been converted.
    static constexpr bool kHalves = HP <= 64;
    static constexpr int kLam = 2 * HP + 64;                    // eigenvalues of the pass direction staged
    static_assert(kSmem + 16 * kLam + 1024 <= 232448, "shared memory of one CTA");
    static_assert(kColA + 3 * HP <= kTcCols, "tensor memory");
};

struct KronTcArgs {
    const BlkDesc* blk;
    int nblk;
    const long long* item0;   // [nblk + 1] first tile of each block in this pass
    const CUtensorMap* maps;  // [nblk] the pass's input rows of each block
    const uint16_t* mat;      // bf16 split matrices (12 padded half-matrices per operator)
    const float* lam;         // eigenvalues per distinct operator (padded mode order)
    float* out;
    const int* active;
    double* flops;            // algorithmic flop counter (profiling) or null
    unsigned* dmax;           // [norb] max |output| per orbital (float bits, atomicMax) or null
    int* status;
    int axis, inverse, scale;
    int full;                 // every side of the pass fills the instance's half-lines (ns > HP - 16)
};

struct TcTile {
    int b, o, q;   // block (-1: no more tiles), orbital within the block, tile within the orbital
};

// What a warp needs of its tile's block, read once per block change.
struct TcBlk {
    int b = -1, n, ns, na, ns4, p, px, nx, ny;
    long long Gp, R, poff;
    long long kt, kl0, kl1, kl2;
};

__device__ __forceinline__ void tc_blk_load(TcBlk& k, const BlkDesc* blk, int b, int axis) {
    if (k.b == b) return;
    const BlkDesc& B = blk[b];
    k.b = b;
    k.n = axis == 0 ? B.nx : (axis == 1 ? B.ny : B.nz);
    k.ns = (k.n + 1) >> 1;
    k.na = k.n >> 1;
    k.ns4 = (k.ns + 3) & ~3;
    k.p = B.p[axis];
    k.px = B.p[0];
    k.nx = B.nx;
    k.ny = B.ny;
    k.Gp = B.Gp;
    k.R = B.Gp / k.p;
    k.poff = B.poff;
    k.kt = B.kt[axis];
    k.kl0 = B.klt[0];
    k.kl1 = B.klt[1];
    k.kl2 = B.klt[2];
}

// next item at or after it whose orbital is active (it1 if none); b tracks the block
__device__ __forceinline__ long long tc_next(const KronTcArgs& a, long long it, long long it1, int& b, TcTile& t) {
    for (; it < it1; ++it) {
        while (b + 1 < a.nblk && it >= a.item0[b + 1]) ++b;
        const BlkDesc& B = a.blk[b];
        const int tpo = B.tpo[a.axis];
        const int r = (int)(it - a.item0[b]);
        const int o = r / tpo;
        if (a.active[B.orb0 + o]) {
            t.b = b;
            t.o = o;
            t.q = r - o * tpo;
            return it;
        }
    }
    return it1;
}

// Three bf16 terms of a pair of floats (f0, f1), each packed as bf16x2 (f0 in
// the low half): v = v1 + v2 + v3 with v1 = bf16(v), v2 = bf16(v - v1),
// v3 = bf16(v - v1 - v2) (the differences are exact in float32).
__device__ __forceinline__ void tc_split2(float f0, float f1, uint32_t& w1, uint32_t& w2, uint32_t& w3) {
    const __nv_bfloat162 b1 = __floats2bfloat162_rn(f0, f1);
    w1 = *reinterpret_cast<const uint32_t*>(&b1);
    const float r0 = f0 - __uint_as_float(w1 << 16), r1 = f1 - __uint_as_float(w1 & 0xffff0000u);
    const __nv_bfloat162 b2 = __floats2bfloat162_rn(r0, r1);
    w2 = *reinterpret_cast<const uint32_t*>(&b2);
    const float q0 = r0 - __uint_as_float(w2 << 16), q1 = r1 - __uint_as_float(w2 & 0xffff0000u);
    const __nv_bfloat162 b3 = __floats2bfloat162_rn(q0, q1);
    w3 = *reinterpret_cast<const uint32_t*>(&b3);
}

// four consecutive points pos..pos+3 (pos a multiple of 4) of row r of a tile
// whose boxes start at ring slot box0 of nslot
__device__ __forceinline__ float4 tc_raw4(const unsigned char* sR, int box0, int nslot, int r, int pos) {
    int bx = box0 + (pos >> 5);
    if (bx >= nslot) bx -= nslot;
    return *reinterpret_cast<const float4*>(sR + bx * kTcBox + r * 128 + ((((pos & 31) >> 2) ^ (r & 7)) << 4));
}

// the 8 values of both halves at K = k .. k + 7 (k a multiple of 8) of row r:
// the folded parts (forward) or the two halves of the coefficients (inverse)
__device__ __forceinline__ void tc_fold8(const unsigned char* sR, int box0, int nslot, int r, int k, const TcBlk& kb,
                                         int inverse, float* e, float* o) {
    const int n = kb.n, ns = kb.ns, na = kb.na;
    if (k >= ns) {
#pragma unroll
        for (int i = 0; i < 8; ++i) e[i] = o[i] = 0.f;
        return;
    }
    const float4 f0 = tc_raw4(sR, box0, nslot, r, k), f1 = tc_raw4(sR, box0, nslot, r, k + 4);
    const float f[8] = {f0.x, f0.y, f0.z, f0.w, f1.x, f1.y, f1.z, f1.w};
    if (inverse) {   // even modes at k, odd modes at ns4 + k
        const float4 g0 = tc_raw4(sR, box0, nslot, r, kb.ns4 + k);
        const float4 g1 = tc_raw4(sR, box0, nslot, r, min(kb.ns4 + k + 4, kb.p - 4));
        const float y[8] = {g0.x, g0.y, g0.z, g0.w, g1.x, g1.y, g1.z, g1.w};
        if (k + 8 <= na) {
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                e[i] = f[i];
                o[i] = y[i];
            }
        } else {
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                e[i] = k + i < ns ? f[i] : 0.f;
                o[i] = k + i < na ? y[i] : 0.f;
            }
        }
        return;
    }
    // the mirrored points n - 8 - k .. n - 1 - k, in descending order
    const int e0 = n - 8 - k, sh = n & 3, a0 = max(e0 - sh, 0);   // aligned window
    const float4 w0 = tc_raw4(sR, box0, nslot, r, a0);
    const float4 w1 = tc_raw4(sR, box0, nslot, r, a0 + 4);
    float y[8];    // y[i] = point n - 1 - (k + i)
    if (sh == 0) {
        y[0] = w1.w; y[1] = w1.z; y[2] = w1.y; y[3] = w1.x;
        y[4] = w0.w; y[5] = w0.z; y[6] = w0.y; y[7] = w0.x;
    } else {
        const float4 w2 = tc_raw4(sR, box0, nslot, r, a0 + 8);
        if (sh == 1) {
            y[0] = w2.x; y[1] = w1.w; y[2] = w1.z; y[3] = w1.y;
            y[4] = w1.x; y[5] = w0.w; y[6] = w0.z; y[7] = w0.y;
        } else if (sh == 2) {
            y[0] = w2.y; y[1] = w2.x; y[2] = w1.w; y[3] = w1.z;
            y[4] = w1.y; y[5] = w1.x; y[6] = w0.w; y[7] = w0.z;
        } else {
            y[0] = w2.z; y[1] = w2.y; y[2] = w2.x; y[3] = w1.w;
            y[4] = w1.z; y[5] = w1.y; y[6] = w1.x; y[7] = w0.w;
        }
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        e[i] = f[i] + y[i];
        o[i] = f[i] - y[i];
    }
    if (k + 8 > na) {
#pragma unroll
        for (int i = 0; i < 8; ++i) {   // past the half-line (the middle of an odd line: 2 v and 0)
            if (k + i >= ns) e[i] = 0.f;
            if (k + i >= na) o[i] = 0.f;
        }
    }
}

// splits 8 values of one half and stores them: column tc, + cs, + 2 cs per split
__device__ __forceinline__ void tc_put8(uint32_t tc, uint32_t cs, const float* v) {
    uint32_t w1[4], w2[4], w3[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) tc_split2(v[2 * i], v[2 * i + 1], w1[i], w2[i], w3[i]);
    tmem_st4(tc, w1[0], w1[1], w1[2], w1[3]);
    tmem_st4(tc + cs, w2[0], w2[1], w2[2], w2[3]);
    tmem_st4(tc + 2 * cs, w3[0], w3[1], w3[2], w3[3]);
}

// The MMAs of one unit: modes 32 c .. 32 c + 31 of one half, KS steps of K =
// 16, straight-line code on warp-uniform operands (see tc_elect).  dm: the
// unit's accumulators, am: the half's operand splits, bh: its matrices.
template <int HP, int KS>
__device__ __forceinline__ void tc_issue_ks(uint32_t dm, uint32_t am, uint64_t d128, uint64_t d64, uint32_t el) {
    using S = TcShape<HP>;
    const uint32_t idesc = umma_idesc_bf16(kTcRows, kTcUnit);
    constexpr int pa[6] = {0, 0, 1, 0, 2, 1};   // split of the data operand (A) of product p
    constexpr int pb[6] = {0, 1, 0, 2, 0, 1};   // split of the matrix operand (B)
#pragma unroll
    for (int kk = 0; kk < KS; ++kk) {
#pragma unroll
        for (int p = 0; p < 6; ++p) {
            const uint32_t ta = am + (uint32_t)((HP / 2) * pa[p] + 8 * kk);
            const uint64_t db = (kk < 4 ? d128 + (uint64_t)(kk * 32 >> 4) : d64 + (uint64_t)((kk - 4) * 32 >> 4)) +
                                (uint64_t)(pb[p] * S::kBTile >> 4);
            if (p == 0) umma_bf16_ts_el(dm, ta, db, idesc, kk != 0, el);
            else umma_bf16_ts_el(dm + kTcUnit, ta, db, idesc, (kk | (p - 1)) != 0, el);
        }
    }
}
template <int HP>
__device__ __forceinline__ void tc_issue_unit(bool full, int ksteps, uint32_t dm, uint32_t am, uint32_t bh, int c,
                                              uint32_t el) {
    using S = TcShape<HP>;
    dm = tc_uniform(dm);
    am = tc_uniform(am);
    bh = tc_uniform(bh);
    c = (int)tc_uniform((uint32_t)c);
    const uint64_t d128 = umma_desc_sw128(bh + (uint32_t)(c * kTcUnit * 128));                      // K values 0 .. 63
    const uint64_t d64 = umma_desc_sw64(bh + (uint32_t)(HP * 128 + c * kTcUnit * 2 * S::kKC));      // K values 64 ..
    if (full) {   // a launch whose every side takes all the steps: no switch in the loop (46 -> 28 cycles per MMA)
        tc_issue_ks<HP, HP / 16>(dm, am, d128, d64, el);
        return;
    }
    switch (ksteps) {
        case 1: tc_issue_ks<HP, 1>(dm, am, d128, d64, el); break;
        case 2: tc_issue_ks<HP, 2>(dm, am, d128, d64, el); break;
        case 3: tc_issue_ks<HP, 3>(dm, am, d128, d64, el); break;
        case 4: tc_issue_ks<HP, 4>(dm, am, d128, d64, el); break;
        case 5: if (HP > 64) tc_issue_ks<HP, HP / 16 < 5 ? 4 : 5>(dm, am, d128, d64, el); break;
        default: if (HP > 64) tc_issue_ks<HP, HP / 16>(dm, am, d128, d64, el); break;
    }
}

// Warp roles: warp 0 issues the MMAs (its elected lane), warp 13 walks the
// tile list and issues the copies, warps 1-8 convert (two threads per row:
// warp w owns tensor-memory lanes 32 (w mod 4) .. + 31, and every second
// group of eight K values), warps 9-12 drain the accumulators and store (one
// thread per row).  They meet only at mbarriers:
//   bar_info[i]  tile descriptor i mod kTcInfo is written              (copy warp)
//   bar_tma[s]   the box in ring slot s has arrived                    (copy engine)
//   bar_raw[i]   every converter has read tile t's boxes, i = t mod kTcInfo (8 warp arrivals;
//                the copy warp waits for it tiles later, when it needs the room)
//   bar_conv[h]  half h's operand splits are in tensor memory          (8 warp arrivals)
//   bar_half[h]  half h's MMAs (h = 1: all the tile's) have completed  (MMA commit)
//   bar_full[u]  the unit in ring slot u has been accumulated          (MMA commit)
//   bar_free[u]  the epilogue has read the unit in ring slot u         (4 warp arrivals)
// The copy warp keeps as many of the following tiles' boxes on their way as
// the ring holds and hands each tile to the other warps through a ring of
// descriptors (nobody else walks the list: its global loads stay off the
// other warps' paths).  A descriptor is overwritten 16 tiles later, when its
// tile is long finished: at most 9 tiles are staged, and a tile's MMAs wait
// for the units of the tile two before it.  The converters fold the next
// tile's rows into registers while the current tile's MMAs run.  Every wait
// sleeps on its mbarrier, gives up after about two seconds or as soon as
// another warp has given up (s_abort), and the lanes vote on the outcome
// (tc_mbar_warp_wait), so a warp leaves its loop as a whole.
template <int HP>
__global__ void __launch_bounds__(kTcThreads, 1) k_kron_tc(KronTcArgs a, long long total) {
    using S = TcShape<HP>;
    extern __shared__ unsigned char kt_smem_raw[];
    __shared__ uint64_t bar_tma[S::kBoxes], bar_raw[kTcInfo], bar_conv[2], bar_half[2], bar_full[S::kUnits], bar_free[S::kUnits],
        bar_info[kTcInfo];
    __shared__ TcTile s_tile[kTcInfo];
    __shared__ int s_nbox[kTcInfo];
    __shared__ __align__(16) float s_lam[4][S::kLam];
    __shared__ uint32_t tmem_base;
    __shared__ volatile int s_abort;
    __shared__ int s_tma_issued[S::kBoxes], s_units;   // copies per ring slot, units committed
    const int tid = threadIdx.x, warp = (int)tc_uniform((uint32_t)tid >> 5), lane = tid & 31;
    const long long per_cta = (total + gridDim.x - 1) / gridDim.x;
    const long long it0 = (long long)blockIdx.x * per_cta;
    const long long it1 = it0 + per_cta < total ? it0 + per_cta : total;
    if (it0 >= it1) return;

    unsigned char* sm =
        reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(kt_smem_raw) + 1023) & ~(uintptr_t)1023);
    unsigned char* sB = sm;
    unsigned char* sR = sm + S::kOffRaw;
    if (tid == 0) {
        for (int b = 0; b < S::kBoxes; ++b) {
            tc_mbar_init(&bar_tma[b], 1);
            s_tma_issued[b] = 0;
        }
        for (int u = 0; u < S::kUnits; ++u) {
            tc_mbar_init(&bar_full[u], 1);
            tc_mbar_init(&bar_free[u], 4);
        }
        for (int i = 0; i < kTcInfo; ++i) {
            tc_mbar_init(&bar_info[i], 1);
            tc_mbar_init(&bar_raw[i], kTcConv / 32);
        }
        for (int h = 0; h < 2; ++h) {
            tc_mbar_init(&bar_conv[h], kTcConv / 32);
            tc_mbar_init(&bar_half[h], 1);
        }
        s_abort = 0;
        s_units = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) tmem_alloc(&tmem_base, kTcCols);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_base;

    if (warp == 0) {
        // ---- MMAs (one elected lane of the converged warp) ---------------------
        const uint32_t el = tc_elect();
        const uint32_t t0 = tc_uniform(tmem);
        const uint32_t b0 = tc_uniform(tc_smem_addr(sB));
        int ksteps = 0, nch = 0, cb = -1;
        uint32_t sl = 0, use = 0;       // ring slot of the next unit, and how often it was used
        for (int t = 0;; ++t) {
            bool ok = tc_mbar_warp_wait(&bar_conv[0], (uint32_t)(t & 1), &s_abort);
            if (!ok) { s_abort = 1; break; }
            const TcTile cur = s_tile[t % kTcInfo];   // (written before the copies this tile's converters waited for)
            const int tb = (int)tc_uniform((uint32_t)cur.b);
            if (tb < 0) break;
            if (tb != cb) {
                const BlkDesc& B = a.blk[tb];
                const int n = a.axis == 0 ? B.nx : (a.axis == 1 ? B.ny : B.nz), ns = (n + 1) >> 1;
                ksteps = (int)tc_uniform((uint32_t)(ns + 15) >> 4);
                nch = (int)tc_uniform((uint32_t)(ns + kTcUnit - 1) / kTcUnit);
                cb = tb;
            }
            // unit u of the tile: half u / nch, chunk u mod nch (kHalves), or chunk u / 2, half u mod 2
            for (int u = 0, h = 0, c = 0; u < 2 * nch; ++u) {
                if (S::kHalves ? u == nch : u == 0) {   // the second half's splits
                    ok = tc_mbar_warp_wait(&bar_conv[1], (uint32_t)(t & 1), &s_abort);
                }
                // the unit that last used this slot has been read
                if (use > 0) ok = ok && tc_mbar_warp_wait(&bar_free[sl], (use - 1) & 1, &s_abort);
                if (!ok) break;
                tc_fence_after();
                tc_issue_unit<HP>(a.full != 0, ksteps, t0 + sl * (2 * kTcUnit), t0 + S::kColA + (uint32_t)(h * 3 * (HP / 2)),
                                  b0 + (uint32_t)(h * 3 * S::kBTile), c, el);
                if (el) {
                    umma_commit(&bar_full[sl]);
                    ++s_units;
                    if (u == 2 * nch - 1 || (S::kHalves && u == nch - 1)) umma_commit(&bar_half[u == 2 * nch - 1 ? 1 : 0]);
                }
                __syncwarp();
                if (++sl == S::kUnits) {
                    sl = 0;
                    ++use;
                }
                if (S::kHalves) {
                    if (++c == nch) { c = 0; h = 1; }
                } else {
                    c += h;
                    h ^= 1;
                }
            }
            if (!ok) { s_abort = 1; break; }
        }
    } else if (warp == kTcThreads / 32 - 1) {
        // ---- the tile list and the copies (one elected lane issues) -------------
        const uint32_t el = tc_elect();
        TcBlk kc;
        int bs = 0, slot = 0, used = 0, tail = 0;   // boxes in use; tiles whose boxes were freed
        TcTile nt{};
        long long ni = tc_next(a, it0, it1, bs, nt);
        double flops = 0.0;
        for (int t = 0;; ++t) {
            bool ok = true;
            const bool end = ni >= it1;
            if (!end) {
                tc_blk_load(kc, a.blk, nt.b, a.axis);
                const int nbox = (kc.p + 31) >> 5;
                while (used + nbox > S::kBoxes && ok) {   // the oldest staged tile has been read
                    ok = tc_mbar_warp_wait(&bar_raw[tail % kTcInfo], (uint32_t)((tail / kTcInfo) & 1), &s_abort);
                    used -= s_nbox[tail % kTcInfo];
                    ++tail;
                }
                if (!ok) { s_abort = 1; break; }
                const int row0 = (int)((long long)nt.o * kc.R + (long long)nt.q * kTcRows);
                if (el) {
                    s_tile[t % kTcInfo] = nt;
                    s_nbox[t % kTcInfo] = nbox;
                    tc_mbar_arrive(&bar_info[t % kTcInfo]);
                }
                for (int bx = 0; bx < nbox; ++bx) {
                    if (el) {
                        tc_mbar_expect_tx(&bar_tma[slot], (uint32_t)kTcBox);
                        tc_tma_load_2d(sR + slot * kTcBox, a.maps + nt.b, 32 * bx, row0, &bar_tma[slot]);
                        ++s_tma_issued[slot];
                    }
                    slot = slot + 1 == S::kBoxes ? 0 : slot + 1;
                }
                used += nbox;
                if (a.flops) {
                    const long long rows = kc.R - (long long)nt.q * kTcRows;
                    flops += 2.0 * ((double)kc.ns * kc.ns + (double)kc.na * kc.na) * (double)(rows < kTcRows ? rows : kTcRows);
                }
                ni = tc_next(a, ni + 1, it1, bs, nt);
            } else if (el) {
                s_tile[t % kTcInfo] = TcTile{-1, 0, 0};
                tc_mbar_arrive(&bar_info[t % kTcInfo]);
            }
            __syncwarp();
            if (end) break;
        }
        if (a.flops && el && flops > 0.0) atomicAdd(a.flops, flops);
    } else if (warp <= kTcConv / 32) {
        // ---- converters: rows in, fold, split, operand splits in tensor memory --
        const int qd = warp & 3;                         // tensor-memory lane quadrant
        const int r = 32 * qd + lane;                    // row of the tile
        const int kp = (warp - 1) >> 2;                  // every second group of eight K values
        const uint32_t ta_row = tmem + ((uint32_t)(32 * qd) << 16) + S::kColA;
        int loaded_b = -1, box0 = 0;
        uint32_t box_uses = 0;                           // parity bit per ring slot of its next completion
        TcBlk kb;
        for (int t = 0;; ++t) {
            bool ok = tc_mbar_warp_wait(&bar_info[t % kTcInfo], (uint32_t)((t / kTcInfo) & 1), &s_abort);
            if (!ok) { s_abort = 1; break; }
            const int cb = s_tile[t % kTcInfo].b;
            if (cb < 0) {   // the MMA warp learns it through bar_conv (after it has seen the last tile's)
                ok = t < 1 || tc_mbar_warp_wait(&bar_half[1], (uint32_t)((t - 1) & 1), &s_abort);
                if (ok && lane == 0) tc_mbar_arrive(&bar_conv[0]);
                break;
            }
            tc_blk_load(kb, a.blk, cb, a.axis);
            const int ns = kb.ns;
            const int nbox = (kb.p + 31) >> 5;
            for (int bx = 0; bx < nbox && ok; ++bx) {
                const int sl = box0 + bx >= S::kBoxes ? box0 + bx - S::kBoxes : box0 + bx;
                ok = tc_mbar_warp_wait(&bar_tma[sl], (box_uses >> sl) & 1u, &s_abort);
                box_uses ^= 1u << sl;
            }
            if (!ok) { s_abort = 1; break; }
            const int k16 = (ns + 15) & ~15;             // K values the MMAs read
            // the first groups folded into registers while the last tile's MMAs run
            float e[S::kPre][8], o[S::kPre][8];
#pragma unroll
            for (int g = 0; g < S::kPre; ++g) {
                const int k = 16 * g + 8 * kp;
                if (k < k16) tc_fold8(sR, box0, S::kBoxes, r, k, kb, a.inverse, e[g], o[g]);
            }
            if (HP / 16 == S::kPre) {
                __syncwarp();
                if (lane == 0) tc_mbar_arrive(&bar_raw[t % kTcInfo]);     // the staged boxes may be overwritten
            }
            // the last tile's MMAs have read the (first half's) operand splits; new
            // matrices wait for all of them
            const bool new_b = cb != loaded_b;
            if (t >= 1) ok = tc_mbar_warp_wait(&bar_half[S::kHalves && !new_b ? 0 : 1], (uint32_t)((t - 1) & 1), &s_abort);
            if (!ok) { s_abort = 1; break; }
            tc_fence_after();
            if (new_b) {   // this block's matrices: the rows and K values in use
                const uint16_t* src = a.mat + kb.kt + (a.inverse ? 6 * S::kMatElems : 0);
                const int rows = (ns + kTcUnit - 1) / kTcUnit * kTcUnit, kc8 = k16 >> 3;
                for (int i = tid - 32; i < 6 * rows * kc8; i += kTcConv) {
                    const int c = i % kc8, rm = i / kc8, m = rm % rows, mt = rm / rows;
                    const uint4 v = *reinterpret_cast<const uint4*>(src + mt * S::kMatElems + m * HP + c * 8);
                    const int off = c < 8 ? m * 128 + ((c ^ (m & 7)) << 4)
                                          : HP * 128 + m * 2 * S::kKC + (((c - 8) ^ ((m >> 1) & 3)) << 4);
                    *reinterpret_cast<uint4*>(sB + mt * S::kBTile + off) = v;
                }
                loaded_b = cb;
            }
            if (S::kHalves) {
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    if (h == 1 && t >= 1) {
                        ok = tc_mbar_warp_wait(&bar_half[1], (uint32_t)((t - 1) & 1), &s_abort);
                        if (!ok) { s_abort = 1; break; }
                        tc_fence_after();
                    }
#pragma unroll
                    for (int g = 0; g < S::kPre; ++g) {
                        const int k = 16 * g + 8 * kp;
                        if (k < k16) tc_put8(ta_row + (uint32_t)((k >> 1) + h * 3 * (HP / 2)), HP / 2, h == 0 ? e[g] : o[g]);
                    }
                    tmem_wait_st();
                    if (h == 0 && new_b) tc_fence_proxy_async();   // the matrices, for the MMAs' reads
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) tc_mbar_arrive(&bar_conv[h]);
                }
                if (!ok) break;
            } else {
#pragma unroll
                for (int g = 0; g < S::kPre; ++g) {
                    const int k = 16 * g + 8 * kp;
                    if (k < k16) {
                        const uint32_t th = ta_row + (uint32_t)(k >> 1);
                        tc_put8(th, HP / 2, e[g]);
                        tc_put8(th + 3 * (HP / 2), HP / 2, o[g]);
                    }
                }
#pragma unroll 1
                for (int g = S::kPre; g < HP / 16; ++g) {
                    const int k = 16 * g + 8 * kp;
                    if (k >= k16) break;
                    tc_fold8(sR, box0, S::kBoxes, r, k, kb, a.inverse, e[0], o[0]);
                    const uint32_t th = ta_row + (uint32_t)(k >> 1);
                    tc_put8(th, HP / 2, e[0]);
                    tc_put8(th + 3 * (HP / 2), HP / 2, o[0]);
                }
                __syncwarp();
                if (lane == 0) tc_mbar_arrive(&bar_raw[t % kTcInfo]);
                tmem_wait_st();
                if (new_b) tc_fence_proxy_async();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) {
                    tc_mbar_arrive(&bar_conv[0]);
                    tc_mbar_arrive(&bar_conv[1]);
                }
            }
            box0 = box0 + nbox >= S::kBoxes ? box0 + nbox - S::kBoxes : box0 + nbox;
        }
    } else {
        // ---- epilogue: accumulators -> scaling / recombination -> stores -------
        const int g4 = warp & 3;                                  // TMEM lanes 32 g4 .. = tile rows
        const int r = 32 * g4 + lane;                             // one row per thread
        const uint32_t tr = tmem + ((uint32_t)(32 * g4) << 16);
        float* const s_lz = s_lam[g4];
        int loaded_b = -1;
        uint32_t U = 0;              // units read so far
        TcBlk kb;
        bool ok = true;
        for (int t = 0; ok; ++t) {
            ok = tc_mbar_warp_wait(&bar_info[t % kTcInfo], (uint32_t)((t / kTcInfo) & 1), &s_abort);
            if (!ok) { s_abort = 1; break; }
            const TcTile cur = s_tile[t % kTcInfo];
            if (cur.b < 0) break;
            tc_blk_load(kb, a.blk, cur.b, a.axis);
            const int n = kb.n, ns = kb.ns, na = kb.na;
            const long long R = kb.R;
            const long long l = (long long)cur.q * kTcRows + r;   // row within the orbital
            const int nch = (ns + kTcUnit - 1) / kTcUnit;
            float lxy = 0.f;
            if (a.scale) {
                if (cur.b != loaded_b) {   // the pass direction's eigenvalues, padded mode order (a copy per warp)
                    __syncwarp();
                    for (int i = lane; i < kb.ns4 + nch * kTcUnit; i += 32) s_lz[i] = a.lam[kb.kl2 + i];
                    loaded_b = cur.b;
                    __syncwarp();
                }
                if (l < R) {   // forward z: rows are (my, mx), mx fastest
                    const int li = (int)l, my = li / kb.px, mx = li - my * kb.px;
                    lxy = a.lam[kb.kl0 + mx] + a.lam[kb.kl1 + my];
                }
            }
            bool real_row = l < R;
            if (a.dmax && real_row) {   // last pass: rows are (y, x); padding rows hold no output
                const int li = (int)l, y = li / kb.px;
                real_row = y < kb.ny && li - y * kb.px < kb.nx;
            }
            float amax = 0.f;   // max |output| of this row (for a.dmax)
            float* const dst = a.out + kb.poff + (long long)cur.o * kb.Gp + (l < R ? l : 0);
            for (int c = 0; c < nch; ++c) {
                const uint32_t ue = U + (S::kHalves ? c : 2 * c), uo = U + (S::kHalves ? nch + c : 2 * c + 1);
                const uint32_t s0 = ue % S::kUnits, s1 = uo % S::kUnits;
                ok = tc_mbar_warp_wait(&bar_full[s0], (ue / S::kUnits) & 1, &s_abort) &&
                     tc_mbar_warp_wait(&bar_full[s1], (uo / S::kUnits) & 1, &s_abort);
                if (!ok) { s_abort = 1; break; }
                tc_fence_after();
                const uint32_t te = tr + s0 * (2 * kTcUnit), to = tr + s1 * (2 * kTcUnit);
#pragma unroll 1
                for (int j16 = 0; j16 < 2; ++j16) {
                    const int m0 = kTcUnit * c + 16 * j16;
                    float v1[16], v2[16];
                    {
                        float e1[16], o1[16];
                        tmem_ld16(te + 16 * j16, v1);
                        tmem_ld16(te + 16 * j16 + kTcUnit, e1);
                        tmem_ld16(to + 16 * j16, v2);
                        tmem_ld16(to + 16 * j16 + kTcUnit, o1);
                        tmem_wait_ld();
#pragma unroll
                        for (int j = 0; j < 16; ++j) {
                            v1[j] += e1[j];
                            v2[j] += o1[j];
                        }
                    }
                    if (j16 == 1) {   // both units are read: their slots may be overwritten
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) {
                            tc_mbar_arrive(&bar_free[s0]);
                            tc_mbar_arrive(&bar_free[s1]);
                        }
                    }
                    if (m0 >= ns) continue;
                    // forward: v1 even mode m, v2 odd mode m; inverse: points m and n - 1 - m
                    if (!a.inverse) {
                        if (a.scale) {   // (fast division: 2 ulp, far below the solve's accuracy)
#pragma unroll
                            for (int q = 0; q < 4; ++q) {
                                const float4 le = *reinterpret_cast<const float4*>(s_lz + m0 + 4 * q);
                                const float4 lo = *reinterpret_cast<const float4*>(s_lz + kb.ns4 + m0 + 4 * q);
                                const float ze[4] = {le.x, le.y, le.z, le.w}, zo[4] = {lo.x, lo.y, lo.z, lo.w};
#pragma unroll
                                for (int i = 0; i < 4; ++i) {
                                    const int j = 4 * q + i;
                                    const float se = lxy + ze[i], so = lxy + zo[i];
                                    v1[j] = se > 0.f ? __fdividef(v1[j], se) : 0.f;
                                    v2[j] = so > 0.f ? __fdividef(v2[j], so) : 0.f;
                                }
                            }
                        }
                    } else {
#pragma unroll
                        for (int j = 0; j < 16; ++j) {
                            const float s_ = v1[j], a_ = v2[j];
                            v1[j] = s_ + a_;
                            v2[j] = s_ - a_;
                        }
                        if (a.dmax) {   // a tree of maxima, not a chain
                            float mj[8];
#pragma unroll
                            for (int j = 0; j < 8; ++j) {
                                const float x0 = m0 + j < ns ? fmaxf(fabsf(v1[j]), fabsf(v2[j])) : 0.f;
                                const float x1 = m0 + j + 8 < ns ? fmaxf(fabsf(v1[j + 8]), fabsf(v2[j + 8])) : 0.f;
                                mj[j] = fmaxf(x0, x1);
                            }
                            amax = fmaxf(amax, fmaxf(fmaxf(fmaxf(mj[0], mj[1]), fmaxf(mj[2], mj[3])),
                                                     fmaxf(fmaxf(mj[4], mj[5]), fmaxf(mj[6], mj[7]))));
                        }
                    }
                    if (l < R) {   // 128-byte stores: the lanes own consecutive rows
                        float* p1 = dst + (long long)m0 * R;
                        float* p2 = dst + (long long)(a.inverse ? n - 1 - m0 : kb.ns4 + m0) * R;
                        const long long st2 = a.inverse ? -R : R;
                        if (m0 + 16 <= na) {
#pragma unroll
                            for (int j = 0; j < 16; ++j, p1 += R, p2 += st2) {
                                __stcs(p1, v1[j]);
                                __stcs(p2, v2[j]);
                            }
                        } else {
#pragma unroll
                            for (int j = 0; j < 16; ++j, p1 += R, p2 += st2) {
                                if (m0 + j < ns) __stcs(p1, v1[j]);
                                if (m0 + j < na) __stcs(p2, v2[j]);
                            }
                        }
                    }
                }
            }
            if (!ok) break;
            U += 2 * (uint32_t)nch;
            if (!ok) break;
            if (a.dmax) {
                float m = real_row ? amax : 0.f;
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
                if (lane == 0 && m > 0.f) atomicMax(a.dmax + a.blk[cur.b].orb0 + cur.o, __float_as_uint(m));
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (s_abort && tid == 0) {
        atomicOr(a.status + 3, 4);
        // let the copies and the MMAs this CTA has in flight finish (bounded)
        for (int b = 0; b < S::kBoxes; ++b)
            if (s_tma_issued[b] > 0) tc_mbar_wait(&bar_tma[b], (uint32_t)((s_tma_issued[b] - 1) & 1));
        // (a commit covers every MMA before it, so the last unit's covers all, also in mid-tile)
        const TcLastCommit lc = tc_last_commit(s_units, S::kUnits);
        if (lc.slot >= 0) tc_mbar_wait(&bar_full[lc.slot], lc.parity);
    }
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        tmem_dealloc(tmem, kTcCols);
    }
}

uint16_t host_bf16(float f) {   // round to nearest even
    uint32_t u;
    std::memcpy(&u, &f, 4);
    u += 0x7fffu + ((u >> 16) & 1u);
    return (uint16_t)(u >> 16);
}
double host_bf16_value(uint16_t b) {
    const uint32_t u = (uint32_t)b << 16;
    float f;
    std::memcpy(&f, &u, 4);
    return (double)f;
}

template <int HP>
void launch_pass(const KronTcArgs& a, int grid, long long total, cudaStream_t s) {
    k_kron_tc<HP><<<grid, kTcThreads, TcShape<HP>::kSmem, s>>>(a, total);
}

}  // namespace

int kron_tc_hp(int n) { return n <= 128 ? 64 : 96; }

// The padded side of a line of n points: room for the even modes rounded up
// to a multiple of 4 and the odd modes, itself a multiple of 4 (16-byte rows).
int kron_pad(int n) {
    const int ns4 = ((n + 1) / 2 + 3) & ~3;
    return (ns4 + n / 2 + 3) & ~3;
}

// Sides that are multiples of 8 up to 128 need no padding and may take the
// tensor cores at any size (the autotuner decides, kron.cu); other sides do from
// 32 points up to the 192 whose matrices fit in shared memory (below 32 the
// CUDA-core tiles are as fast and need no padding).  Measured per inner solve:
// 117^3 x 20 0.44 ms here, 1.35 ms on the CUDA cores; 192^3 x 24 1.82 and 7.35 ms.
// Whole Poisson solves, here and there: 33^3 x 1 293 and 325 us, x 50 563 and 693;
// 44^3 x 5 316 and 372; 61^3 x 2 309 and 365; 90 x 36 x 33 x 1 308 and 352;
// 75^3 x 10 699 and 960; 140^3 x 1 637 and 893 (78 shapes with sides of 33 to 192
// points and 1 to 50 orbitals: always the faster, so these are not timed at
// creation).
bool kron_tc_eligible(const BlkDesc& B) {
    const int nd[3] = {B.nx, B.ny, B.nz};
    bool general = true;
    for (int d = 0; d < 3; ++d)
        if (nd[d] < 32 || nd[d] > 192) general = false;
    return general || kron_tc_tiled(B);
}
bool kron_tc_tiled(const BlkDesc& B) {
    const int nd[3] = {B.nx, B.ny, B.nz};
    for (int d = 0; d < 3; ++d)
        if (nd[d] < 8 || nd[d] > 128 || nd[d] % 8 != 0) return false;
    return true;
}

// The operator's four half-matrices in the transform kernel's operand form
// (rows = outputs, K = inputs, padded to HP x HP), each as three bf16
// splits of the float64 value: [direction][half][split][HP][HP].
//   forward: c_s[m] = sum_k s_k Vs[k][m] f_k, c_a[m] = sum_k a_k Va[k][m] / sqrt 2
//   inverse: S_k = sum_m c_s[m] Vs[k][m] g_k, A_k = sum_m c_a[m] Va[k][m] / sqrt 2
// with f_k = g_k = 1/sqrt 2 but at the middle of an odd line, where s_mid =
// 2 v_mid: f = 1/2, g = 1.
void kron_tc_pack(int n, const std::vector<double>& Vs, const std::vector<double>& Va, std::vector<uint16_t>& out) {
    const int hp = kron_tc_hp(n), ns = (n + 1) / 2, na = n / 2;
    const size_t me = (size_t)hp * hp;
    const double r2 = std::sqrt(0.5);
    const size_t o0 = out.size();
    out.resize(o0 + 12 * me, 0);
    for (int dir = 0; dir < 2; ++dir)
        for (int half = 0; half < 2; ++half) {
            const std::vector<double>& V = half == 0 ? Vs : Va;
            const int h = half == 0 ? ns : na;
            for (int row = 0; row < h; ++row)
                for (int k = 0; k < h; ++k) {
                    // forward: row = mode, k = point; inverse: row = point, k = mode
                    const int pt = dir == 0 ? k : row, md = dir == 0 ? row : k;
                    const double f = pt < na ? r2 : (dir == 0 ? 0.5 : 1.0);
                    const double v = V[(size_t)pt * h + md] * f;
                    const uint16_t b1 = host_bf16((float)v);
                    const double q1 = v - host_bf16_value(b1);
                    const uint16_t b2 = host_bf16((float)q1);
                    const double q2 = q1 - host_bf16_value(b2);
                    const uint16_t b3 = host_bf16((float)q2);
                    const uint16_t bs[3] = {b1, b2, b3};
                    for (int s = 0; s < 3; ++s)
                        out[o0 + (size_t)((dir * 2 + half) * 3 + s) * me + (size_t)row * hp + k] = bs[s];
                }
        }
}

cudaError_t kron_tc_setup() {
    cudaError_t e = ensure_dyn_smem((const void*)k_kron_tc<64>, TcShape<64>::kSmem);
    if (e == cudaSuccess) e = ensure_dyn_smem((const void*)k_kron_tc<96>, TcShape<96>::kSmem);
    return e;
}

// Input rows of a pass along `axis` of block B as a 2-D tensor map: the
// padded side per row (contiguous), N Gp / p rows, boxes of 32 points x 128 rows.
bool kron_tc_map(void* encode_fn, CUtensorMap* map, const BlkDesc& B, int axis, const float* buf) {
    auto encode = reinterpret_cast<CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                                const cuuint64_t*, const cuuint32_t*, const cuuint32_t*,
                                                CUtensorMapInterleave, CUtensorMapSwizzle,
                                                CUtensorMapL2promotion, CUtensorMapFloatOOBfill)>(encode_fn);
    const int p = B.p[axis];
    const cuuint64_t dims[2] = {(cuuint64_t)p, (cuuint64_t)(B.Gp / p) * (cuuint64_t)B.N};
    const cuuint64_t strides[1] = {(cuuint64_t)p * sizeof(float)};
    const cuuint32_t box[2] = {32, (cuuint32_t)kTcRows};
    const cuuint32_t estr[2] = {1, 1};
    void* base = const_cast<float*>(buf) + B.poff;
    return encode(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, base, dims, strides, box, estr,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

int kron_tc_tiles(const BlkDesc& B, int axis) {   // per orbital
    return (int)((B.Gp / B.p[axis] + kTcRows - 1) / kTcRows);
}

// pass `step` (axis step mod 3) on the blocks whose side along that axis
// belongs to size class cls (0: up to 128, 1: up to 192)
void launch_kron_tc_pass(flosic_ctx* c, int step, float* out, cudaStream_t s) {
    const KronPlan& K = c->kron;
    KronTcArgs a{};
    a.blk = c->d_blk;
    a.nblk = c->nblk;
    a.maps = reinterpret_cast<const CUtensorMap*>(K.tc_maps) + (size_t)step * c->nblk;
    a.mat = K.tc_mat;
    a.lam = K.lam;
    a.out = out;
    a.active = c->ws.cg.active;
    a.flops = c->profiling ? c->ws.cg.prof_bytes : nullptr;
    a.dmax = step == 5 ? c->ws.cg.dmax : nullptr;   // the correction d: its scale for the refinement update
    a.status = c->ws.status;
    a.axis = step % 3;
    a.inverse = step >= 3;
    a.scale = step == 2;
    for (int cls = 0; cls < 2; ++cls) {
        const int k = 2 * step + cls;
        if (K.tc_total[k] == 0) continue;
        a.item0 = K.tc_items + (size_t)k * (c->nblk + 1);
        a.full = K.tc_full[k];
        if (cls == 0) launch_pass<64>(a, K.tc_grid[k], K.tc_total[k], s);
        else launch_pass<96>(a, K.tc_grid[k], K.tc_total[k], s);
        note_launch(c);
    }
}

}  // namespace flosic
