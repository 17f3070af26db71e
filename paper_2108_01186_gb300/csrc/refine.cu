// Mixed-precision refinement of the per-orbital Poisson solves (Sec. II.A
// solves them iteratively; splitting the precision is this library's).
//
// The float32 multigrid-preconditioned CG computes corrections d of
// A d = r.  The solution x, the right-hand side b and the residual
// r = b - A x live in unevaluated float-float pairs (hi, lo), about 48
// significant bits: Knuth's error-free two-sum for additions and an
// FMA-based exact two-product.  GB300 runs float64 at a small fraction of
// its float32 rate, so inside the refinement loop no float64 operation runs
// per grid point; float64 appears only where x is joined into the float64
// result (one addition per point).  b arrives in pairs from the
// right-hand-side pass; a warm start is split with integer operations.
//
// Round structure per orbital:  r = b - A x (pairs) -> stop if
// r.r <= tol^2 b.b, else a float32 solve of A d = float(r) to
// max(inner_tol^2 r.r, tol^2 b.b / 4) -> x += d (pairs).
#include <cmath>
#include <vector>

#include <cudaTypedefs.h>

#include "ffsweep.cuh"
#include "ixsweep.cuh"
#include "tcgen05.cuh"

namespace flosic {


// Last CTA of an orbital, once r.r is known: the outer stop test, else the
// start of the next float32 solve (its target, active flag and counters).
__device__ __forceinline__ void start_round(CgState& st, int o, double rr, double tol2, double inner_tol2,
                                            int max_iter) {
    st.rr[o] = rr;
    st.active[o] = 0;
    if (!(rr > tol2 * st.bb[o])) {
        st.oactive[o] = 0;
        st.conv[o] = 1;
        atomicSub(st.n_oactive, 1);
        return;
    }
    if (st.iters[o] >= max_iter || !isfinite(rr)) {
        st.oactive[o] = 0;
        atomicSub(st.n_oactive, 1);
        return;
    }
    const double a = inner_tol2 * rr, c = 0.25 * tol2 * st.bb[o];
    st.thr[o] = a > c ? a : c;
    st.rz[o] = 0.0;
    st.beta[o] = 0.0;
    st.active[o] = 1;
    atomicAdd(st.n_active, 1);
}

// Start of the refinement: b arrives in pairs (from the right-hand-side
// pass), x = warm start (pairs) or 0; b.b per orbital.  Without a warm start
// the residual is b itself: r32 = float(b), d32 = 0 (p32 = r32 when given)
// and the first float32 solve starts here.  keep_zero (cold start of a solver
// that overwrites d, the Kronecker solve): neither x nor d is stored; xz marks
// x as zero until the first update writes it.
__global__ void __launch_bounds__(256) k_ff_init(const BlkDesc* __restrict__ blk, const LvlDesc* __restrict__ L,
                                                 const int4* __restrict__ tiles, const int* __restrict__ orb_blk,
                                                 const float2* __restrict__ b, const double* __restrict__ V,
                                                 float2* __restrict__ x, float* __restrict__ r32,
                                                 float* __restrict__ p32, float* __restrict__ d32, int warm,
                                                 int keep_zero, double tol2, double inner_tol2, int max_iter,
                                                 CgState st) {
    __shared__ double scratch[32];
    const TilePos P = tile_pos(blk, L, tiles, orb_blk, blockIdx.x);
    if (!st.oactive[P.o]) return;
    const LvlDesc& D = L[P.b];
    const BlkDesc& B = blk[P.b];
    const int io = P.o - B.orb0;
    float bb = 0.f;
    tile_rows<float>(D, P, [&](int px, int py, int pz, long long g, int n) {
        const long long q = pad_index(B, io, px, py, pz);   // in r32 (and p32, d32)
        if (n == 4) {   // aligned group of four points: 16-byte accesses
            const float4 b01 = *reinterpret_cast<const float4*>(b + g);       // pairs g, g+1
            const float4 b23 = *reinterpret_cast<const float4*>(b + g + 2);   // pairs g+2, g+3
            const float4 bh = make_float4(b01.x, b01.z, b23.x, b23.z);
            bb += bh.x * bh.x + bh.y * bh.y + bh.z * bh.z + bh.w * bh.w;
            if (warm) {
                const double2 v01 = *reinterpret_cast<const double2*>(V + g);
                const double2 v23 = *reinterpret_cast<const double2*>(V + g + 2);
                const float2 a = d2ff(v01.x), c = d2ff(v01.y), e = d2ff(v23.x), f = d2ff(v23.y);
                *reinterpret_cast<float4*>(x + g) = make_float4(a.x, a.y, c.x, c.y);
                *reinterpret_cast<float4*>(x + g + 2) = make_float4(e.x, e.y, f.x, f.y);
            } else {
                const float4 z4 = make_float4(0.f, 0.f, 0.f, 0.f);
                if (!keep_zero) {
                    *reinterpret_cast<float4*>(x + g) = z4;
                    *reinterpret_cast<float4*>(x + g + 2) = z4;
                    *reinterpret_cast<float4*>(d32 + q) = z4;
                }
                *reinterpret_cast<float4*>(r32 + q) = bh;
                if (p32) *reinterpret_cast<float4*>(p32 + q) = bh;
            }
            return;
        }
        for (int k = 0; k < n; ++k) {
            const float bh = b[g + k].x;
            bb += bh * bh;
            if (warm) {
                x[g + k] = d2ff(V[g + k]);
            } else {
                if (!keep_zero) {
                    x[g + k] = make_float2(0.f, 0.f);
                    d32[q + k] = 0.f;
                }
                r32[q + k] = bh;
                if (p32) p32[q + k] = bh;
            }
        }
    }, !warm || aligned16(V));
    if (tile_arrive(bb, st.part, blockIdx.x, st.count + P.o, D.ntile, scratch)) {
        const double sum = tile_gather(st.part, P.first, D.ntile, scratch);
        if (linear_tid() == 0) {
            st.count[P.o] = 0;
            st.bb[P.o] = sum;
            st.xz[P.o] = (!warm && keep_zero) ? 1 : 0;
            if (!warm) start_round(st, P.o, sum, tol2, inner_tol2, max_iter);
        }
    }
}

// r = b - A x in pairs on the tiles of the float-float sweep.  Writes
// r32 = float(r), d32 = 0 (p32 = r32 when given) and starts the next round;
// with store_r also r itself as pairs over b (each point's r needs only its
// own b), for the rounds that then update r from the corrections.
__global__ void __launch_bounds__(256) k_residual12_ff(const BlkDesc* __restrict__ blk, const LvlDesc* __restrict__ L,
                                                       const int4* __restrict__ tiles, const int* __restrict__ orb_blk,
                                                       float2* __restrict__ b, const float2* __restrict__ x,
                                                       float* __restrict__ r32, float* __restrict__ p32,
                                                       float* __restrict__ d32, double tol2, double inner_tol2,
                                                       int max_iter, int store_r, CgState st) {
    __shared__ ff plane[kPY][kPX];
    __shared__ double scratch[32];
    const TilePos P = tile_pos(blk, L, tiles, orb_blk, blockIdx.x);
    if (!st.oactive[P.o]) return;
    const LvlDesc& D = L[P.b];
    const ff ih2 = to_ff(d2ff(1.0 / (D.h * D.h)));   // once per CTA
    const BlkDesc& B = blk[P.b];
    // the thread's columns in r32, p32, d32 (a division per point to find them from g
    // took 12 % of a warm solve of 150^3 x 4)
    const int io = P.o - B.orb0, cx = P.x0 + threadIdx.x, cy = P.y0 + threadIdx.y;
    const long long dsz = (long long)B.p[0] * B.p[1];
    const long long qc[2] = {pad_index(B, io, cx, cy, 0), pad_index(B, io, cx, cy + kTileY / 2, 0)};
    float rrf = 0.f;
    ff_sweep12(
        D, P, [&](long long g) { return x[g]; },
        [&](long long g, int k, int z, ff, ff acc) {
            // acc = h^2 Delta_h x, so r = b - A x = b + acc / h^2
            const ff r = ff_add(to_ff(b[g]), ff_mul(acc, ih2));
            const float rv = r.h;
            if (store_r) b[g] = make_float2(r.h, r.l);
            const long long q = qc[k] + z * dsz;
            r32[q] = rv;
            d32[q] = 0.f;
            if (p32) p32[q] = rv;
            rrf += rv * rv;
        },
        plane);
    if (tile_arrive(rrf, st.part, blockIdx.x, st.count + P.o, D.ntile, scratch)) {
        const double sum = tile_gather(st.part, P.first, D.ntile, scratch);
        if (linear_tid() == 0) {
            st.count[P.o] = 0;
            start_round(st, P.o, sum, tol2, inner_tol2, max_iter);
        }
    }
}

// ---------------------------------------------------------------------------
// Exact stencil sums for the refinement update (weights W_m: ixsweep.cuh).
// A float32 field d whose magnitude is below 2^e splits exactly into
// y = d 2^(28-e) = hi + lo with hi = rint(y) an integer (|hi| <= 2^28) and
// |lo| <= 1/2: the hi parts are summed and weighted in integers, so that
// part is exact, and the lo parts in float32, an error of a few units
// of 2^(e-28) / 831600 in h^2 Delta_h d per point -- about 1e-14 of
// max |d| / h^2, below the float-float sweep's error on smooth fields.
// ---------------------------------------------------------------------------
// Two neighbouring points' parts, the low ones side by side for packed
// two-lane additions.
struct __align__(16) IxPair {
    int h0, h1;      // rint(y) of either point
    float2 l;        // y - rint(y)
};

// y = d 2^es (exact) split into hi + lo, for sums taken in unsigned (wrapping)
// integers: a non-finite y carries inf / NaN in lo, so it reaches the
// residual, and its saturated integer part only wraps the integer sum.
__device__ __forceinline__ IxPair ix_split_w(float2 d, float s) {
    const float y0 = d.x * s, y1 = d.y * s;
    const float r0 = rintf(y0), r1 = rintf(y1);
    return {__float2int_rn(r0), __float2int_rn(r1), make_float2(y0 - r0, y1 - r1)};
}

// Per orbital, max |d| over its grid (float bits in st.dmax, atomicMax on
// the bit patterns of non-negative floats); the update's last CTA of the
// orbital resets it.  NaN values are skipped here and reach the residual
// through the split.
__global__ void __launch_bounds__(256) k_dmax(const BlkDesc* __restrict__ blk, const LvlDesc* __restrict__ L,
                                              const int4* __restrict__ tiles, const int* __restrict__ orb_blk,
                                              const float* __restrict__ d32, CgState st) {
    const TilePos P = tile_pos(blk, L, tiles, orb_blk, blockIdx.x);
    if (!st.oactive[P.o]) return;
    const LvlDesc& D = L[P.b];
    const BlkDesc& B = blk[P.b];
    if (B.tc) return;   // recorded by the tensor-core transforms
    const int io = P.o - B.orb0;
    float m = 0.f;
    tile_rows<float>(D, P, [&](int px, int py, int pz, long long, int n) {
        const long long g = pad_index(B, io, px, py, pz);
        if (n == 4) {
            const float4 v = *reinterpret_cast<const float4*>(d32 + g);
            m = fmaxf(m, fmaxf(fmaxf(fabsf(v.x), fabsf(v.y)), fmaxf(fabsf(v.z), fabsf(v.w))));
            return;
        }
        for (int k = 0; k < n; ++k) m = fmaxf(m, fabsf(d32[g + k]));
    });
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((linear_tid() & 31) == 0 && m > 0.f) atomicMax(st.dmax + P.o, __float_as_uint(m));
}

// Scales of the update of an orbital with max |d| (float bits): |d| < 2^(E -
// 126) with E the biased exponent of max |d|, so y = d 2^es with es = 154 - E
// (kept within the normal range) has |y| < 2^28; is = 2^-es, and cf turns the
// weighted sums into Delta_h d.
struct IxScale {
    float sc, is;
    ff cf;
};
__device__ __forceinline__ IxScale ix_scale(unsigned dmax, double h) {
    const int E = (int)((dmax >> 23) & 0xffu);
    const int es = max(-126, min(126, 154 - E));
    return {__uint_as_float((unsigned)(es + 127) << 23), __uint_as_float((unsigned)(127 - es) << 23),
            to_ff(d2ff(ldexp(1.0 / ((double)kW12Den * h * h), -es)))};
}

// The weighted sums (integer and float parts) of a pair of points: pc its
// entry in the split plane of kPitch pairs, q its z-window with plane z - 6 in
// slot u.  The low parts of the two points run as packed two-lane operations
// (the x-neighbours at odd distances are not pairs: two plain additions).
template <int kPitch>
__device__ __forceinline__ void ix_sums2(const IxPair* pc, const IxPair (&q)[kQ], int u, long long& I0, long long& I1,
                                         float2& Lo) {
    constexpr int kWc = (int)w12_centre3();
    constexpr int kW[kHalf + 1] = {kWc,           (int)w12_int(1), (int)w12_int(2), (int)w12_int(3),
                                   (int)w12_int(4), (int)w12_int(5), (int)w12_int(6)};
    IxPair xw[kHalf + 1];   // columns -6 .. 7 of the row
#pragma unroll
    for (int k2 = 0; k2 < kHalf + 1; ++k2) xw[k2] = pc[k2 - kHalf / 2];
    auto xh = [&](int c) { return (unsigned)((c & 1) ? xw[c >> 1].h1 : xw[c >> 1].h0); };
    auto xl = [&](int c) { return (c & 1) ? xw[c >> 1].l.y : xw[c >> 1].l.x; };
    const IxPair c = q[u + kHalf];
    I0 = (long long)kW[0] * c.h0;
    I1 = (long long)kW[0] * c.h1;
    Lo = __fmul2_rn(make_float2((float)kW[0], (float)kW[0]), c.l);
#pragma unroll
    for (int m = 1; m <= kHalf; ++m) {
        const IxPair uu = pc[-m * kPitch], ww = pc[m * kPitch];   // rows -+ m
        const IxPair a = q[u + kHalf - m], b = q[u + kHalf + m];
        const unsigned h0 = ((xh(kHalf - m) + xh(kHalf + m)) + ((unsigned)uu.h0 + (unsigned)ww.h0)) +
                            ((unsigned)a.h0 + (unsigned)b.h0);
        const unsigned h1 = ((xh(kHalf + 1 - m) + xh(kHalf + 1 + m)) + ((unsigned)uu.h1 + (unsigned)ww.h1)) +
                            ((unsigned)a.h1 + (unsigned)b.h1);
        const float2 x2 = (m & 1) ? make_float2(xl(kHalf - m) + xl(kHalf + m), xl(kHalf + 1 - m) + xl(kHalf + 1 + m))
                                  : __fadd2_rn(xw[(kHalf - m) >> 1].l, xw[(kHalf + m) >> 1].l);
        const float2 l = __fadd2_rn(__fadd2_rn(x2, __fadd2_rn(uu.l, ww.l)), __fadd2_rn(a.l, b.l));
        I0 += (long long)kW[m] * (int)h0;
        I1 += (long long)kW[m] * (int)h1;
        Lo = __ffma2_rn(make_float2((float)kW[m], (float)kW[m]), l, Lo);
    }
}

// r + Delta_h d (pairs) of a point from its weighted sums, and d there (exact)
__device__ __forceinline__ ff ix_update(long long I, float Lo, ff cf, float2 r) {
    return ff_add(to_ff(r), ff_mul(ix_to_ff_b(I, Lo), cf));
}
__device__ __forceinline__ float2 ix_centre(IxPair c, float is) {
    return make_float2((__int2float_rn(c.h0) + c.l.x) * is, (__int2float_rn(c.h1) + c.l.y) * is);
}
__device__ __forceinline__ ff ix_add(float2 x, float d) {   // x + d
    const ff s = ff_two_sum(x.x, d);
    return ff_quick(s.h, s.l + x.y);
}

// One refinement round's update from the float32 correction d of the inner
// solve: r -= A d (r in pairs, in place: r_{k+1} = b - A x_{k+1} =
// r_k - A d_k), x += d (pairs), r32 = float(r), and the next round's start.
// A d comes from the exact integer sums above, on the tiles of the other
// 12th-order sweeps (a CTA owns a 32 x 16 column tile and marches along z).
// d is left as it is (neighbouring tiles read it as halo): this serves inner
// solvers that overwrite d (the Kronecker-product solve), not those that
// start from d = 0.  kXZ: the first update after a cold start that stored no
// x (x = 0, not read).
//
// This form has its operands staged by the copy engine (blocks whose rows and
// offset are 16-byte aligned and that have no periodic direction: the zero fill
// of the copies is the zero ghost value).  A ring of kURing stages runs ahead of
// the z-march, each holding the plane z of d with its halo (48 x 28: x0 - 8
// keeps the copy 16-byte aligned), d at plane z + 6 (32 x 16, the head of the
// register z-queues) and r and x at plane z (32 x 16 pairs).  Each plane's d is
// split once into shared memory
// (hi, lo; two buffers, so one barrier per plane serves both the split plane
// and the stage of the plane before); a thread owns the two points (x0 + 2 tx +
// a, y0 + ty), reads their x-window (14 values) and y-windows as 16-byte pairs
// and keeps their z-windows in registers.
// What bounds it: instruction issue and shared-memory traffic.  With the parts
// of a point pair side by side (16-byte splits and stores, packed low-part sums)
// Poisson solves of 128^3 x 64 take 6.93 -> 6.71 ms, 192^3 x 24 8.94 -> 8.66.
constexpr int kUX = 48;                              // staged width: x0 - 8 .. x0 + 39
constexpr int kUY = kTileY + 2 * kHalf;              // 28: y0 - 6 .. y0 + 21
constexpr int kUPlane = kUX * kUY;                   // floats of the halo plane
constexpr int kUCtr = kTileX * kTileY;               // points of a centre tile
constexpr int kUStage = kUPlane + 5 * kUCtr;         // floats: plane, d head, r pairs, x pairs
constexpr int kURing = 5;
constexpr unsigned kUStageBytes = 4u * kUStage;

// the stages, two split planes (one barrier per plane), the stages' mbarriers
size_t update_tma_smem() { return 4 * (size_t)kURing * kUStage + sizeof(IxPair) * kUPlane + 8 * kURing + 128; }

template <bool kXZ>
__global__ void __launch_bounds__(256, 2) k_update12_tma(const BlkDesc* __restrict__ blk, const LvlDesc* __restrict__ L,
                                                         const int4* __restrict__ tiles, const int* __restrict__ orb_blk,
                                                         const CUtensorMap* __restrict__ maps,
                                                         const float* __restrict__ d32, float2* __restrict__ r,
                                                         float2* __restrict__ x, float* __restrict__ r32,
                                                         double tol2, double inner_tol2, int max_iter, CgState st,
                                                         int* __restrict__ status) {
    extern __shared__ __align__(128) unsigned char us_raw[];
    unsigned char* smem = us_raw + ((128 - (tc_smem_addr(us_raw) & 127)) & 127);
    float* ring = reinterpret_cast<float*>(smem);
    IxPair* spb = reinterpret_cast<IxPair*>(smem + 4 * (size_t)kURing * kUStage);   // two split planes
    uint64_t* bar = reinterpret_cast<uint64_t*>(smem + 4 * (size_t)kURing * kUStage + sizeof(IxPair) * kUPlane);
    __shared__ double scratch[32];
    const TilePos P = tile_pos(blk, L, tiles, orb_blk, blockIdx.x);
    if (!st.oactive[P.o] || !L[P.b].utma) return;
    const LvlDesc& D = L[P.b];
    const CUtensorMap* mp = maps + 4 * P.b;   // d with halo, d centre, r pairs, x pairs
    const int oi = P.o - blk[P.b].orb0;
    const int tid = threadIdx.y * blockDim.x + threadIdx.x;
    const int nzt = P.z1 - P.z0;
    constexpr bool xz = kXZ;   // x is zero and not stored yet: its tiles are not copied
    __shared__ IxScale s_scale;   // one thread's float64 division
    if (tid == 0) s_scale = ix_scale(st.dmax[P.o], D.h);
    auto issue = [&](int k) {
        uint64_t* b = bar + (k % kURing);
        float* sg = ring + (size_t)(k % kURing) * kUStage;
        const int zz = P.z0 + k;
        tc_mbar_expect_tx(b, xz ? kUStageBytes - 8u * kUCtr : kUStageBytes);
        tc_tma_load_4d(sg, mp + 0, P.x0 - 8, P.y0 - kHalf, zz, oi, b);
        tc_tma_load_4d(sg + kUPlane, mp + 1, P.x0, P.y0, zz + kHalf, oi, b);
        tc_tma_load_4d(sg + kUPlane + kUCtr, mp + 2, 2 * P.x0, P.y0, zz, oi, b);
        if (!xz) tc_tma_load_4d(sg + kUPlane + 3 * kUCtr, mp + 3, 2 * P.x0, P.y0, zz, oi, b);
    };
    if (tid == 0) {
        for (int k = 0; k < kURing; ++k) tc_mbar_init(bar + k, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        for (int k = 0; k < kURing && k < nzt; ++k) issue(k);
    }
    __syncthreads();
    const float sc = s_scale.sc, is = s_scale.is;
    const ff cf = s_scale.cf;
    const int tx = threadIdx.x, ty = threadIdx.y;   // 16 x 16
    const int gx = P.x0 + 2 * tx, gy = P.y0 + ty;
    const bool in = gx < D.nx && gy < D.ny;           // nx is even: gx + 1 < nx as well
    const long long sy = D.nx, sz = (long long)D.nx * D.ny;
    const long long col = gy * sy + gx;
    // d and r32 hold the block with padded sides
    const BlkDesc& B = blk[P.b];
    const long long dsz = (long long)B.p[0] * B.p[1];
    const long long dcol = B.poff + (long long)oi * B.Gp + (long long)gy * B.p[0] + gx;
    // z-windows of the two points: plane z - 6 + j of step k0 + u in slot u + j
    IxPair q[kQ];
#pragma unroll
    for (int j = 0; j < 2 * kHalf; ++j) {
        const int zz = P.z0 - kHalf + j;
        float2 v = make_float2(0.f, 0.f);
        if (in && zz >= 0 && zz < D.nz) v = *reinterpret_cast<const float2*>(d32 + zz * dsz + dcol);
        q[j] = ix_split_w(v, sc);
    }
    float rrf = 0.f;
    const int pc = (ty + kHalf) * (kUX / 2) + tx + 4;   // the points' pair in the staged plane
    for (int k0 = 0; k0 < nzt; k0 += kZU) {
#pragma unroll
        for (int u = 0; u < kZU; ++u) {
            const int k = k0 + u;
            if (k >= nzt) break;
            if (!tc_mbar_wait(bar + (k % kURing), (uint32_t)((k / kURing) & 1))) atomicOr(status + 3, 8);
            const float* sg = ring + (size_t)(k % kURing) * kUStage;
            IxPair* const sp = spb + (k & 1) * (kUPlane / 2);
            for (int e = tid; e < kUPlane / 2; e += 256) sp[e] = ix_split_w(reinterpret_cast<const float2*>(sg)[e], sc);
            q[u + 2 * kHalf] =
                ix_split_w(*reinterpret_cast<const float2*>(sg + kUPlane + ty * kTileX + 2 * tx), sc);
            // the split plane is written, and every thread has finished plane k - 1: its
            // stage takes plane k - 1 + kURing (the other split plane is free for plane k + 1)
            __syncthreads();
            if (tid == 0 && k >= 1 && k - 1 + kURing < nzt) {
                tc_fence_proxy_async();
                issue(k - 1 + kURing);
            }
            long long I0, I1;
            float2 Lo;
            ix_sums2<kUX / 2>(sp + pc, q, u, I0, I1, Lo);
            if (in) {
                const float4 rv = *reinterpret_cast<const float4*>(sg + kUPlane + kUCtr + ty * 2 * kTileX + 4 * tx);
                const float4 xv = xz ? make_float4(0.f, 0.f, 0.f, 0.f)
                                     : *reinterpret_cast<const float4*>(sg + kUPlane + 3 * kUCtr + ty * 2 * kTileX + 4 * tx);
                const long long g = P.base + (P.z0 + k) * sz + col;
                const ff rn[2] = {ix_update(I0, Lo.x, cf, make_float2(rv.x, rv.y)), ix_update(I1, Lo.y, cf, make_float2(rv.z, rv.w))};
                const float2 dc = ix_centre(q[u + kHalf], is);
                const ff xn[2] = {ix_add(make_float2(xv.x, xv.y), dc.x), ix_add(make_float2(xv.z, xv.w), dc.y)};
                rrf += rn[0].h * rn[0].h;
                rrf += rn[1].h * rn[1].h;
                *reinterpret_cast<float4*>(r + g) = make_float4(rn[0].h, rn[0].l, rn[1].h, rn[1].l);
                *reinterpret_cast<float4*>(x + g) = make_float4(xn[0].h, xn[0].l, xn[1].h, xn[1].l);
                *reinterpret_cast<float2*>(r32 + (P.z0 + k) * dsz + dcol) = make_float2(rn[0].h, rn[1].h);
            }
        }
        ix_shift(q);
    }
    if (tile_arrive(rrf, st.part, blockIdx.x, st.count + P.o, D.ntile, scratch)) {
        const double sum = tile_gather(st.part, P.first, D.ntile, scratch);
        if (linear_tid() == 0) {
            st.count[P.o] = 0;
            st.dmax[P.o] = 0u;
            st.xz[P.o] = 0;
            start_round(st, P.o, sum, tol2, inner_tol2, max_iter);
        }
    }
}

// The same update for the other blocks (odd rows, rows or offsets off 16
// bytes, periodic directions).  d's planes arrive by asynchronous copies
// (IxStage), r and V by 8-byte copies one plane ahead; one barrier per plane.
// x is the caller's float64 V itself, V += d: a conversion and one float64
// addition per point, and no pass joins pairs into V at the end (117^3 x 20
// 2.60 -> 2.44 ms, an uneven batch 6.40 -> 6.06 ms).  k_update12_tma keeps pairs:
// with V its two launches at 128^3 x 64 grew by more than the 0.35 ms of the join.
// What bounds it: instruction issue, as above.  The plain-load sweep it
// replaced (two barriers per plane, 24 eight-byte shared loads per point, its
// z-windows moved every plane) took 1149 us for the two updates of 117^3 x 20,
// this one about 1000 us.
constexpr int kCOffRx = kIxPts * 8 * kIxRing;
constexpr int kCSmem = kCOffRx + 2 * 16 * kUCtr;     // two stages of r and V

template <bool kXZ>
__global__ void __launch_bounds__(256, 2) k_update12_cp(const BlkDesc* __restrict__ blk, const LvlDesc* __restrict__ L,
                                                        const int4* __restrict__ tiles, const int* __restrict__ orb_blk,
                                                        const float* __restrict__ d32, float2* __restrict__ r,
                                                        double* __restrict__ V, float* __restrict__ r32, double tol2,
                                                        double inner_tol2, int max_iter, CgState st) {
    extern __shared__ __align__(16) unsigned char uc_raw[];
    IxPair* const ring = reinterpret_cast<IxPair*>(uc_raw);
    float2* const rx = reinterpret_cast<float2*>(uc_raw + kCOffRx);   // [2][r pairs, V][kUCtr]
    __shared__ double scratch[32];
    const TilePos P = tile_pos(blk, L, tiles, orb_blk, blockIdx.x);
    if (!st.oactive[P.o] || L[P.b].utma) return;
    const LvlDesc& D = L[P.b];
    const BlkDesc& B = blk[P.b];
    const int tid = threadIdx.y * blockDim.x + threadIdx.x;
    const int nx = D.nx, ny = D.ny, nz = D.nz, per = D.per;
    __shared__ IxScale s_scale;   // one thread's float64 division
    if (tid == 0) s_scale = ix_scale(st.dmax[P.o], D.h);
    const long long sy = nx, sz = (long long)nx * ny;
    // d and r32 hold the block with padded sides
    const int dpx = B.p[0];
    const long long dsz = (long long)dpx * B.p[1], db = B.poff + (long long)(P.o - B.orb0) * B.Gp;
    IxStage sg;
    sg.init(D, P, dpx, tid);
    const bool vec = (dpx & 1) == 0 && (db & 1) == 0 && (per & 1) == 0;
    const int nzt = P.z1 - P.z0;
    auto copy_d = [&](int k, int slot) {   // plane z0 + k
        int z = P.z0 + k;
        if (per & 4) z = wrap_coord(z, nz);
        const bool okz = z < nz;
        const float* pl = d32 + db + (okz ? z * dsz : 0);
#pragma unroll
        for (int j = 0; j < kIxU; ++j)
            if (sg.wants(j, k < nzt)) sg.copy(j, ring + slot * kIxPairs + tid + j * 256, pl, okz, vec, nx);
    };
    auto split = [&](int k, int slot, float sc) {
#pragma unroll
        for (int j = 0; j < kIxU; ++j)
            if (sg.wants(j, k < nzt)) {
                IxPair* const at = ring + slot * kIxPairs + tid + j * 256;
                *at = ix_split_w(*reinterpret_cast<const float2*>(at), sc);
            }
    };
    // r and V of plane z0 + k: rows of 32 points per warp
    const int cxp = P.x0 + (tid & 31), cyp = P.y0 + (tid >> 5);
    auto copy_rx = [&](int k) {
        float2* const dst = rx + (k & 1) * 2 * kUCtr + tid;
        const long long g0 = P.base + (P.z0 + k) * sz;
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const bool ok = cxp < nx && cyp + 8 * j < ny;
            const long long g = g0 + (ok ? (cyp + 8 * j) * sy + cxp : 0);
            cp_async<8>(dst + 256 * j, r + g, ok ? 8 : 0);
            if (!kXZ) cp_async<8>(dst + kUCtr + 256 * j, V + g, ok ? 8 : 0);
        }
    };
    for (int k = 0; k < kHalf; ++k) copy_d(k, k);
    copy_rx(0);
    cp_async_commit();
    copy_d(kHalf, kHalf);
    cp_async_commit();
    copy_d(kHalf + 1, kHalf + 1);
    cp_async_commit();

    const int tx = threadIdx.x, ty = threadIdx.y;     // 16 x 16; points (x0 + 2 tx + a, y0 + ty)
    const int gx = P.x0 + 2 * tx, gy = P.y0 + ty;
    const bool in0 = gx < nx && gy < ny, in1 = gx + 1 < nx && gy < ny;
    const long long col = gy * sy + gx, dcol = db + (long long)gy * dpx + gx;
    const int ctr = (ty + kHalf) * (kPX / 2) + tx + kHalf / 2;   // the pair in a staged plane
    __syncthreads();
    const float sc = s_scale.sc, is = s_scale.is;
    const ff cf = s_scale.cf;
    IxPair q[kQ];   // z-windows: step k0 + u's in slots u .. u + 12
#pragma unroll
    for (int j = 0; j < kHalf; ++j) {   // planes z0 - 6 .. z0 - 1 straight from memory
        int z = P.z0 - kHalf + j;
        if (per & 4) z = wrap_coord(z, nz);
        const float* pl = d32 + z * dsz + dcol;
        const bool okz = z >= 0 && z < nz;
        q[j] = ix_split_w(make_float2(okz && in0 ? pl[0] : 0.f, okz && in1 ? pl[1] : 0.f), sc);
    }
    asm volatile("cp.async.wait_group 2;" ::: "memory");
    for (int k = 0; k < kHalf; ++k) split(k, k, sc);
    __syncthreads();
#pragma unroll
    for (int k = 0; k < kHalf; ++k) q[kHalf + k] = ring[k * kIxPairs + ctr];
    float rrf = 0.f;
    int slot = 0;   // of plane z0 + k
    for (int k0 = 0; k0 < nzt; k0 += kZU) {
#pragma unroll
        for (int u = 0; u < kZU; ++u) {
            const int k = k0 + u;
            if (k >= nzt) break;
            // the slot of plane k + 8 held plane k - 2, which every thread has finished; all
            // but that copy have arrived (the planes up to k + 7, plane k's r and V)
            if (k + 2 < nzt) copy_d(k + kHalf + 2, ix_slot(slot, kHalf + 2));
            cp_async_commit();
            asm volatile("cp.async.wait_group 1;" ::: "memory");
            const int hslot = ix_slot(slot, kHalf);
            split(k + kHalf, hslot, sc);
            // plane k + 6 is split, and every thread has finished plane k - 1, whose stage of
            // r and V takes plane k + 1's
            __syncthreads();
            if (k + 1 < nzt) copy_rx(k + 1);
            cp_async_commit();
            q[u + 2 * kHalf] = ring[hslot * kIxPairs + ctr];
            const IxPair* const pc = ring + slot * kIxPairs + ctr;
            slot = ix_slot(slot, 1);
            long long I0, I1;
            float2 Lo;
            ix_sums2<kPX / 2>(pc, q, u, I0, I1, Lo);
            const float2* const st2 = rx + (k & 1) * 2 * kUCtr + ty * kTileX + 2 * tx;
            const float4 rv = *reinterpret_cast<const float4*>(st2);
            const ff rn[2] = {ix_update(I0, Lo.x, cf, make_float2(rv.x, rv.y)), ix_update(I1, Lo.y, cf, make_float2(rv.z, rv.w))};
            const float2 dc = ix_centre(q[u + kHalf], is);
            double2 vn = make_double2(f2d(dc.x), f2d(dc.y));
            if (!kXZ) {
                const double2 vo = *reinterpret_cast<const double2*>(st2 + kUCtr);
                vn.x += vo.x;
                vn.y += vo.y;
            }
            const int z = P.z0 + k;
            const long long g = P.base + z * sz + col;
            if (in0) {
                r[g] = make_float2(rn[0].h, rn[0].l);
                V[g] = vn.x;
                r32[z * dsz + dcol] = rn[0].h;
                rrf += rn[0].h * rn[0].h;
            }
            if (in1) {
                r[g + 1] = make_float2(rn[1].h, rn[1].l);
                V[g + 1] = vn.y;
                r32[z * dsz + dcol + 1] = rn[1].h;
                rrf += rn[1].h * rn[1].h;
            }
        }
        ix_shift(q);
    }
    if (tile_arrive(rrf, st.part, blockIdx.x, st.count + P.o, D.ntile, scratch)) {
        const double sum = tile_gather(st.part, P.first, D.ntile, scratch);
        if (linear_tid() == 0) {
            st.count[P.o] = 0;
            st.dmax[P.o] = 0u;   // every CTA of the orbital has read it (and xz)
            st.xz[P.o] = 0;      // V is stored now
            start_round(st, P.o, sum, tol2, inner_tol2, max_iter);
        }
    }
}

// The float-float weights, after checking the update's integer weights
// against the float64 ones (a mismatch fails the context's creation), and the
// shared memory of the update that needs no tensor maps.
cudaError_t upload_ff_weights() {
    if (!ix_weights_match()) return cudaErrorInvalidValue;
    cudaError_t e = ensure_dyn_smem((const void*)k_update12_cp<false>, kCSmem);
    if (e == cudaSuccess) e = ensure_dyn_smem((const void*)k_update12_cp<true>, kCSmem);
    if (e != cudaSuccess) return e;
    return upload_ffsweep_weights();
}

// Tensor maps of the update's operands, four per block, each a 4-D view
// (x, y, z, orbital): d with 48 x 28 boxes and 32 x 16 boxes, and the pair
// arrays r (b) and x as float32 rows of 2 nx values with 64 x 16 boxes.
// Blocks with a periodic direction, or whose rows or offset are not
// 16-byte aligned, take k_update12_cp (flag utma = 0).  Returns the number
// of blocks on the copy-engine path.
int setup_update_maps(flosic_ctx* c) {
    void* fn = nullptr;
    cudaDriverEntryPointQueryResult q{};
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess || !fn)
        return 0;
    auto encode = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(fn);
    std::vector<CUtensorMap> maps(4 * (size_t)c->nblk);
    std::vector<LvlDesc>& L0 = c->mg.h_lvl[0];
    int n_ok = 0;
    for (int b = 0; b < c->nblk; ++b) {
        const BlkDesc& B = c->blk[b];
        L0[b].utma = 0;
        if (B.p[0] % 4 != 0 || B.poff % 4 != 0 || B.nx % 2 != 0 || B.off % 2 != 0 || B.per != 0) continue;
        const cuuint64_t dims[4] = {(cuuint64_t)B.nx, (cuuint64_t)B.ny, (cuuint64_t)B.nz, (cuuint64_t)B.N};
        const cuuint64_t strides[3] = {(cuuint64_t)B.p[0] * 4, (cuuint64_t)B.p[0] * B.p[1] * 4, (cuuint64_t)B.Gp * 4};
        const cuuint64_t dims2[4] = {2 * (cuuint64_t)B.nx, (cuuint64_t)B.ny, (cuuint64_t)B.nz, (cuuint64_t)B.N};
        const cuuint64_t strides2[3] = {(cuuint64_t)B.nx * 8, (cuuint64_t)B.nx * B.ny * 8, (cuuint64_t)B.G * 8};
        const cuuint32_t box_halo[4] = {(cuuint32_t)kUX, (cuuint32_t)kUY, 1, 1};
        const cuuint32_t box_ctr[4] = {(cuuint32_t)kTileX, (cuuint32_t)kTileY, 1, 1};
        const cuuint32_t box_pair[4] = {2 * (cuuint32_t)kTileX, (cuuint32_t)kTileY, 1, 1};
        const cuuint32_t estr[4] = {1, 1, 1, 1};
        float* d = c->ws.d32 + B.poff;
        float* rb = reinterpret_cast<float*>(c->ws.b64 + B.off);
        float* xb = reinterpret_cast<float*>(c->ws.r64 + B.off);
        bool ok = true;
        auto enc = [&](CUtensorMap* m, void* base, const cuuint64_t* dm, const cuuint64_t* sd, const cuuint32_t* bx) {
            return encode(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, base, dm, sd, bx, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                          CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                          CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
        };
        ok = enc(&maps[4 * b + 0], d, dims, strides, box_halo) && enc(&maps[4 * b + 1], d, dims, strides, box_ctr) &&
             enc(&maps[4 * b + 2], rb, dims2, strides2, box_pair) && enc(&maps[4 * b + 3], xb, dims2, strides2, box_pair);
        if (!ok) continue;
        L0[b].utma = 1;
        ++n_ok;
    }
    if (n_ok == 0) return 0;
    void* dm = nullptr;
    if (cudaMalloc(&dm, sizeof(CUtensorMap) * maps.size()) != cudaSuccess) return 0;
    c->allocations.push_back(dm);
    if (cudaMemcpy(dm, maps.data(), sizeof(CUtensorMap) * maps.size(), cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaFuncSetAttribute((const void*)k_update12_tma<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)update_tma_smem()) != cudaSuccess ||
        cudaFuncSetAttribute((const void*)k_update12_tma<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)update_tma_smem()) != cudaSuccess ||
        cudaMemcpy(c->mg.d_lvl[0], L0.data(), sizeof(LvlDesc) * c->nblk, cudaMemcpyHostToDevice) != cudaSuccess) {
        for (auto& D : L0) D.utma = 0;
        cudaMemcpy(c->mg.d_lvl[0], L0.data(), sizeof(LvlDesc) * c->nblk, cudaMemcpyHostToDevice);
        return 0;
    }
    c->d_umaps = dm;
    return n_ok;
}

// x += d32 in pairs for the orbitals still refining.
__global__ void __launch_bounds__(256) k_correct_ff(const BlkDesc* __restrict__ blk, const LvlDesc* __restrict__ L,
                                                    const int4* __restrict__ tiles, const int* __restrict__ orb_blk,
                                                    const float* __restrict__ d32, float2* __restrict__ x,
                                                    CgState st) {
    const TilePos P = tile_pos(blk, L, tiles, orb_blk, blockIdx.x);
    if (!st.oactive[P.o]) return;
    const LvlDesc& D = L[P.b];
    tile_elementwise<float>(D, P, [&](long long g, int n) {
        if (n == 4) {
            const float4 d = *reinterpret_cast<const float4*>(d32 + g);
            float4 a = *reinterpret_cast<float4*>(x + g);       // pairs g, g+1
            float4 c = *reinterpret_cast<float4*>(x + g + 2);   // pairs g+2, g+3
            ff s;
            s = ff_two_sum(a.x, d.x); s = ff_quick(s.h, s.l + a.y); a.x = s.h; a.y = s.l;
            s = ff_two_sum(a.z, d.y); s = ff_quick(s.h, s.l + a.w); a.z = s.h; a.w = s.l;
            s = ff_two_sum(c.x, d.z); s = ff_quick(s.h, s.l + c.y); c.x = s.h; c.y = s.l;
            s = ff_two_sum(c.z, d.w); s = ff_quick(s.h, s.l + c.w); c.z = s.h; c.w = s.l;
            *reinterpret_cast<float4*>(x + g) = a;
            *reinterpret_cast<float4*>(x + g + 2) = c;
        } else {
            const float2 v = x[g];
            ff s = ff_two_sum(v.x, d32[g]);
            s = ff_quick(s.h, s.l + v.y);
            x[g] = make_float2(s.h, s.l);
        }
    });
}

// V = 0 for the orbitals of k_update12_cp's blocks that it never updated (no solve needed).
__global__ void __launch_bounds__(256) k_zero_unsolved(const BlkDesc* __restrict__ blk, const LvlDesc* __restrict__ L,
                                                       const int* __restrict__ orb_blk, const int* __restrict__ xz,
                                                       double* __restrict__ V) {
    const int o = blockIdx.x, b = orb_blk[o];
    if (!xz[o] || L[b].utma) return;
    const BlkDesc& B = blk[b];
    double* v = V + B.off + (long long)(o - B.orb0) * B.G;
    for (long long g = (long long)blockIdx.y * 256 + threadIdx.x; g < B.G; g += 256LL * gridDim.y) v[g] = 0.0;
}

// V = x (pairs joined into float64), every orbital (utma: of the blocks of k_update12_tma).
__global__ void __launch_bounds__(256) k_join_ff(const BlkDesc* __restrict__ blk, const LvlDesc* __restrict__ L,
                                                 const int4* __restrict__ tiles, const int* __restrict__ orb_blk,
                                                 const float2* __restrict__ x, const int* __restrict__ xz,
                                                 int utma, double* __restrict__ V) {
    const TilePos P = tile_pos(blk, L, tiles, orb_blk, blockIdx.x);
    const LvlDesc& D = L[P.b];
    if (utma && !D.utma) return;
    if (xz[P.o]) {   // never updated (no solve needed): V = 0
        tile_elementwise<float>(D, P, [&](long long g, int n) {
            for (int k = 0; k < n; ++k) V[g + k] = 0.0;
        });
        return;
    }
    tile_elementwise<float>(D, P, [&](long long g, int n) {
        if (n == 4) {   // aligned group of four points: 16-byte accesses
            const float4 a = *reinterpret_cast<const float4*>(x + g);
            const float4 c = *reinterpret_cast<const float4*>(x + g + 2);
            *reinterpret_cast<double2*>(V + g) = make_double2(ff2d(make_float2(a.x, a.y)), ff2d(make_float2(a.z, a.w)));
            *reinterpret_cast<double2*>(V + g + 2) =
                make_double2(ff2d(make_float2(c.x, c.y)), ff2d(make_float2(c.z, c.w)));
            return;
        }
        for (int k = 0; k < n; ++k) V[g + k] = ff2d(x[g + k]);
    }, aligned16(V));
}

static dim3 tile_threads() { return dim3(kTileX, kTileY / 2); }

// x is the solution in pairs (float2 per point), p32 may be null.
void launch_ff_init(flosic_ctx* c, const double* b, const double* V, bool warm, bool keep_zero, float2* x,
                    float* p32, double tol2, double inner_tol2, cudaStream_t s) {
    const Multigrid& M = c->mg;
    k_ff_init<<<(unsigned)M.ntiles[0], tile_threads(), 0, s>>>(
        c->d_blk, M.d_lvl[0], M.d_tiles[0], c->d_orb_blk, reinterpret_cast<const float2*>(b), V, x, c->ws.r32, p32,
        c->ws.d32, warm ? 1 : 0, keep_zero ? 1 : 0, tol2, inner_tol2, c->opt.max_iter, c->ws.cg);
    note_launch(c);
}

void launch_residual_ff(flosic_ctx* c, const double* b, const float2* x, float* p32, double tol2,
                        double inner_tol2, bool store_r, cudaStream_t s) {
    const Multigrid& M = c->mg;
    k_residual12_ff<<<(unsigned)M.ntiles[0], tile_threads(), 0, s>>>(
        c->d_blk, M.d_lvl[0], M.d_tiles[0], c->d_orb_blk, reinterpret_cast<float2*>(const_cast<double*>(b)), x,
        c->ws.r32, p32, c->ws.d32, tol2, inner_tol2, c->opt.max_iter, store_r ? 1 : 0, c->ws.cg);
    note_launch(c);
}

// x_zero: the first update after a cold start that stored no x
void launch_update_ff(flosic_ctx* c, double* r, float2* x, double* V, bool x_zero, double tol2, double inner_tol2,
                      cudaStream_t s) {
    const Multigrid& M = c->mg;
    if (c->kron.n_simt > 0) {   // the tensor-core passes record max |d| themselves
        k_dmax<<<(unsigned)M.ntiles[0], tile_threads(), 0, s>>>(c->d_blk, M.d_lvl[0], M.d_tiles[0], c->d_orb_blk,
                                                                c->ws.d32, c->ws.cg);
        note_launch(c);
    }
    if (c->n_utma_blocks > 0) {   // blocks whose operands the copy engine stages
        auto kern = x_zero ? k_update12_tma<true> : k_update12_tma<false>;
        kern<<<(unsigned)M.ntiles[0], dim3(kTileX / 2, kTileY), update_tma_smem(), s>>>(
            c->d_blk, M.d_lvl[0], M.d_tiles[0], c->d_orb_blk, (const CUtensorMap*)c->d_umaps, c->ws.d32,
            reinterpret_cast<float2*>(r), x, c->ws.r32, tol2, inner_tol2, c->opt.max_iter, c->ws.cg, c->ws.status);
        note_launch(c);
    }
    if (c->n_utma_blocks < c->nblk) {   // the rest: asynchronous copies, x = V
        auto kern = x_zero ? k_update12_cp<true> : k_update12_cp<false>;
        kern<<<(unsigned)M.ntiles[0], dim3(kTileX / 2, kTileY), kCSmem, s>>>(
            c->d_blk, M.d_lvl[0], M.d_tiles[0], c->d_orb_blk, c->ws.d32, reinterpret_cast<float2*>(r), V, c->ws.r32,
            tol2, inner_tol2, c->opt.max_iter, c->ws.cg);
        note_launch(c);
    }
}

void launch_correct_ff(flosic_ctx* c, float2* x, cudaStream_t s) {
    const Multigrid& M = c->mg;
    k_correct_ff<<<(unsigned)M.ntiles[0], tile_threads(), 0, s>>>(c->d_blk, M.d_lvl[0], M.d_tiles[0], c->d_orb_blk,
                                                                  c->ws.d32, x, c->ws.cg);
    note_launch(c);
}

// After the rounds: V = x.  The Kronecker rounds (kron) of k_update12_cp's blocks left V
// complete but for orbitals never updated from a cold start.
void launch_join_ff(flosic_ctx* c, const float2* x, bool kron, bool warm, double* V, cudaStream_t s) {
    const Multigrid& M = c->mg;
    if (!kron || c->n_utma_blocks > 0) {
        k_join_ff<<<(unsigned)M.ntiles[0], tile_threads(), 0, s>>>(c->d_blk, M.d_lvl[0], M.d_tiles[0], c->d_orb_blk, x,
                                                                   c->ws.cg.xz, kron ? 1 : 0, V);
        note_launch(c);
    }
    if (kron && !warm && c->n_utma_blocks < c->nblk) {
        k_zero_unsolved<<<dim3(c->norb, 16), 256, 0, s>>>(c->d_blk, M.d_lvl[0], c->d_orb_blk, c->ws.cg.xz, V);
        note_launch(c);
    }
}

}  // namespace flosic
