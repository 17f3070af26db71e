// SC_AvgSIC Hamiltonian apply (Sec. II.C, Eq. 13): the averaged SIC
// potential enters one Kohn-Sham Hamiltonian per spin,
//   H psi_a = -1/2 Delta_h psi_a + (v_loc + V_avg,sigma) psi_a,
// with the same 12th-order Laplacian and zero Dirichlet boundary as the
// Poisson solves (orbitals vanish outside the box).  v_loc stands for the
// remaining local terms of Eq. 13 (external, Hartree, v_xc), one field per
// system; V_avg is the averaged SIC potential of the energy pass (already
// scaled by s), one field per spin block.  Either may be absent.
#include "ixsweep.cuh"

namespace flosic {

__constant__ double c_w64[kHalf + 1];   // this file's copy of the 12th-order weights

// ---------------------------------------------------------------------------
// Mixed precision: psi as a top digit and a float32 pair, their stencil sums
// free of rounding but in the pairs' low parts.
//
// A tile's psi (with the halo its taps reach) lies below 2^k, k from the
// tiles' largest exponents (k_tile_exp); it is scaled to lie below 2^100.  A
// value splits into v = b 2^89 + (h + l): b an integer of at most 2^11, h + l the
// rest as a float32 pair.  The b's of the six neighbours at a distance and their
// weighting are integer sums; the h's are summed by error-free two-sums and
// weighted by exact products; l's, two-sum and product errors are added in
// float32.  So what is lost is 2^-48 of each value (the pair's own resolution,
// any size of value) and never more than 2^-60 of the tile's largest: a field's
// tail keeps the bits that a fixed point would take from it, and its bulk is
// as exact as float64.  (Two digits of 29 bits below the tile's largest value, the
// former kernel, held 85 % of this library's orbitals on 128^3 points, the tails, in fewer
// bits than a pair does, a quarter of them as zero.)
//
// What bounds it: instruction issue and latencies at 16 warps per SM (477
// instructions per point, 61 % of the issue slots).  A value is split once, when its plane arrives (IxStage); one
// barrier per plane.  The planes z - 6 .. z - 1 of a thread's points are in registers,
// z + 1 .. z + 6 in the ring.  Float64 operations cost most (an SM does two per cycle): the
// join of the sums and the potential take two per point (six: 3.32 ms).  128^3 x 64
// orbitals with both potentials 2.73 ms, of which k_tile_exp 0.15: the float-float
// sweep with plain loads took 5.81, the two digits 2.21.  Error against 64 bits in the 2-norm
// (96^3, Gaussians): 1.3e-13, 2.1e-15 with the digits, 1.7e-15 now.
// ---------------------------------------------------------------------------
constexpr int kHRing = 9;                            // staged planes: see the z-loop
constexpr int kHOffTop = kIxPts * 8 * kHRing;        // the top digits, behind the pairs
constexpr int kHSmem = kHOffTop + kIxPts * 2 * kHRing;
constexpr int kExpBad = 1 << 16;                     // a tile with a value beyond 2^799, an infinity or a NaN
constexpr int kExpMin = 300, kExpMax = 1821;         // scale exponents in use: the results stay normal float64
__device__ __forceinline__ int expo(double v) { return (__double2hiint(v) >> 20) & 0x7ff; }

// Per tile: the largest biased exponent of its psi, + kExpBad.  With both potentials
// the tiles of a block's first orbital also add them up (vsum, a field per block), so that
// the sweep loads and adds one field for every orbital.
__global__ void __launch_bounds__(256) k_tile_exp(const BlkDesc* __restrict__ blk, const LvlDesc* __restrict__ L,
                                                  const int4* __restrict__ tiles, const int* __restrict__ orb_blk,
                                                  const double* __restrict__ psi, const double* __restrict__ vloc,
                                                  const double* __restrict__ vavg, double* __restrict__ vsum,
                                                  int* __restrict__ texp) {
    __shared__ int s_max, s_bad;
    const TilePos P = tile_pos(blk, L, tiles, orb_blk, blockIdx.x);
    const BlkDesc& B = blk[P.b];
    if (vloc && vavg && P.o == B.orb0)
        tile_elementwise<float>(L[P.b], P, [&](long long g, int n) {
            for (int k = 0; k < n; ++k) {
                const long long q = g - P.base + k;
                vsum[B.voff + q] = vloc[B.soff + q] + vavg[B.voff + q];
            }
        });
    if (linear_tid() == 0) s_max = s_bad = 0;
    const bool al = (reinterpret_cast<uintptr_t>(psi) & 15) == 0;
    int m = 0, bad = 0;
    auto take = [&](double v) {
        const int e = expo(v);
        if (e > kExpMax) bad = kExpBad;
        else m = max(m, e);
    };
    tile_elementwise<float>(L[P.b], P, [&](long long g, int n) {
        if (n == 4 && al) {
            const double2 a = *reinterpret_cast<const double2*>(psi + g), b = *reinterpret_cast<const double2*>(psi + g + 2);
            take(a.x); take(a.y); take(b.x); take(b.y);
        } else {
            for (int k = 0; k < n; ++k) take(psi[g + k]);
        }
    });
    m = (int)__reduce_max_sync(0xffffffffu, (unsigned)m);
    bad = (int)__reduce_or_sync(0xffffffffu, (unsigned)bad);
    __syncthreads();   // s_max, s_bad are set
    if ((linear_tid() & 31) == 0) {
        atomicMax(&s_max, m);
        if (bad) s_bad = bad;
    }
    __syncthreads();
    if (linear_tid() == 0) texp[blockIdx.x] = s_max | s_bad;
}

// Two neighbouring points' parts: pairs h + l, and the top digits as unsigned
// 16-bit lanes b + kTopBias (the weights of a point's 37 taps sum to zero, so the
// bias leaves no trace, and six lanes add up without a carry).
struct __align__(16) HPair {
    float2 h, l;
};
constexpr float kTopUnit = 6.18970019642690137e26f;   // 2^89
constexpr int kTopBias = 4096;

__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __ffma2_rn(b, make_float2(-1.f, -1.f), a); }
// a + b = s + e exactly, one lane and two at once
__device__ __forceinline__ float two_sum(float a, float b, float& e) {
    const ff s = ff_two_sum(a, b);
    e = s.l;
    return s.h;
}
__device__ __forceinline__ float2 two_sum2(float2 a, float2 b, float2& e) {
    const float2 s = __fadd2_rn(a, b), bb = sub2(s, a);
    e = __fadd2_rn(sub2(a, sub2(s, bb)), sub2(b, bb));
    return s;
}

// One value v 2^(1122 - et) (below 2^100 by its tile's et): f its sign, power of two and
// the 21 leading bits, pw the power of two alone; the 32 bits below as two floats, v = f +
// (a 2^16 + b) 2^-52 pw.  Integer operations: a 64-bit conversion would run on the float64
// pipe.  Zero where v exceeds et (the staged corners, which no tap reads, and
// the values that make a tile bad) or is below 2^-173 of it.
__device__ __forceinline__ void top_parts(double v, unsigned lo, float& f, float& pw, float& a, float& b) {
    const unsigned hw = (unsigned)__double2hiint(v), lw = (unsigned)__double2loint(v);
    const unsigned d = (hw & 0x7fffffffu) - lo;
    const unsigned w = d < (174u << 20) ? ((d << 3) + (53u << 23)) | (hw & 0x80000000u) : 0u;
    f = __uint_as_float(w);
    pw = __uint_as_float(w & 0xff800000u);
    a = __uint_as_float(__byte_perm(lw, 0x4B000000u, 0x7632)) - 8388608.f;
    b = __uint_as_float(__byte_perm(lw, 0x4B000000u, 0x7610)) - 8388608.f;
}
// lo: the least high word in use, (et - 173) 2^20
__device__ __forceinline__ HPair top_split(double2 v, unsigned lo, unsigned& top) {
    float2 f, pw, a, b;
    top_parts(v.x, lo, f.x, pw.x, a.x, b.x);
    top_parts(v.y, lo, f.y, pw.y, a.y, b.y);
    constexpr float kM = kTopUnit * (float)(0xC00000 + kTopBias);   // f + kM rounds f to the units of the top digit
    constexpr float k36 = 1.f / 68719476736.f, k16 = 1.f / 65536.f;
    const float2 m2 = make_float2(kM, kM);
    const float2 tq = __fadd2_rn(f, m2);
    top = __byte_perm(__float_as_uint(tq.x), __float_as_uint(tq.y), 0x5410);
    const float2 r1 = sub2(f, sub2(tq, m2));                       // exact, 0 or larger than t
    const float2 u = __fmul2_rn(pw, make_float2(k36, k36)), t = __fmul2_rn(a, u);
    HPair p;
    p.h = __fadd2_rn(r1, t);
    p.l = __ffma2_rn(b, __fmul2_rn(u, make_float2(k16, k16)), sub2(t, sub2(p.h, r1)));
    return p;
}
// f 2^off in float64, exactly (off keeps it normal; float32 subnormals become 0)
__device__ __forceinline__ double f2d_scaled(float f, int off) {
    const unsigned b = __float_as_uint(f), e = (b >> 23) & 0xffu, m = b & 0x7fffffu;
    const unsigned hi = e == 0 ? 0u : (b & 0x80000000u) | ((e + 896u + (unsigned)off) << 20) | (m >> 3);
    return __hiloint2double((int)hi, (int)(m << 29));
}
// (I 2^89 + h + l) c 2^off of two points (|I| < 2^37): the sum as a normalised pair (48 bits
// of the Laplacian itself), its product with the pair c, one float64 addition each.  (With
// the sum and the product in float64, four operations a point: 3.32 against 3.03 ms.)
__device__ __forceinline__ void top_join(long long I0, long long I1, float2 h, float2 l, ff c, int off, double* r) {
    // I = a 2^14 + b, both exact floats and neither larger than I's terms
    const int a0 = (int)((I0 + 8192) >> 14), a1 = (int)((I1 + 8192) >> 14);
    auto f = [](int k) { return __int_as_float(0x4B400000 + k) - 12582912.f; };   // |k| < 2^22
    const float2 a = make_float2(f(a0), f(a1)), b = make_float2(f((int)I0 - (a0 << 14)), f((int)I1 - (a1 << 14)));
    const float2 ka = make_float2(kTopUnit * 16384.f, kTopUnit * 16384.f), kb = make_float2(kTopUnit, kTopUnit);
    float2 e1, e2;
    const float2 y = two_sum2(__fmul2_rn(b, kb), h, e1);
    const float2 s = two_sum2(__fmul2_rn(a, ka), y, e2);
    const float2 t = __fadd2_rn(__fadd2_rn(e1, e2), l);
    const float2 sh = __fadd2_rn(s, t), sl = sub2(t, sub2(sh, s));
    const float2 ch = make_float2(c.h, c.h), cl = make_float2(c.l, c.l);
    const float2 ph = __fmul2_rn(sh, ch);
    const float2 pl = __ffma2_rn(sl, ch, __ffma2_rn(sh, cl, __ffma2_rn(sh, ch, make_float2(-ph.x, -ph.y))));
    r[0] = f2d_scaled(ph.x, off) + f2d_scaled(pl.x, off);
    r[1] = f2d_scaled(ph.y, off) + f2d_scaled(pl.y, off);
}

__global__ void __launch_bounds__(256, 2) k_hamiltonian_mixed(const BlkDesc* __restrict__ blk, const LvlDesc* __restrict__ L,
                                                              const int4* __restrict__ tiles,
                                                              const int* __restrict__ orb_blk,
                                                              const double* __restrict__ psi,
                                                              const double* __restrict__ v, int per_system,
                                                              const int* __restrict__ texp, double* __restrict__ hpsi) {
    extern __shared__ __align__(16) unsigned char hs_raw[];
    HPair* const ring = reinterpret_cast<HPair*>(hs_raw);
    unsigned* const tops = reinterpret_cast<unsigned*>(hs_raw + kHOffTop);
    __shared__ int s_exp, s_bad;
    __shared__ ff s_cf;
    __shared__ int s_off;
    const TilePos P = tile_pos(blk, L, tiles, orb_blk, blockIdx.x);
    const LvlDesc& D = L[P.b];
    const BlkDesc& B = blk[P.b];
    const int tid = threadIdx.y * 16 + threadIdx.x;
    const int nx = D.nx, ny = D.ny, nz = D.nz, per = D.per;
    if (tid == 0) {
        s_exp = kExpMin;
        s_bad = 0;
    }
    __syncthreads();
    if (tid < 1 + 12 * 3) {   // the largest exponent in this tile (thread 0) and in those of the six points on either side
        int c[3] = {P.x0, P.y0, P.z0};
        const int n3[3] = {nx, ny, nz}, end[3] = {min(P.x0 + kTileX, nx), min(P.y0 + kTileY, ny), P.z1};
        bool ok = true;
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            const int j = tid - 1 - 12 * d;
            if (j >= 0 && j < 12) {
                c[d] = j < kHalf ? c[d] - kHalf + j : end[d] + j - kHalf;
                if (per & (1 << d)) c[d] = wrap_coord(c[d], n3[d]);
                ok = c[d] >= 0 && c[d] < n3[d];
            }
        }
        if (ok) {
            const int ntx = (nx + kTileX - 1) / kTileX, nty = (ny + kTileY - 1) / kTileY;
            const int e = texp[P.first + ((long long)(c[2] / D.tz) * nty + c[1] / kTileY) * ntx + c[0] / kTileX];
            atomicMax(&s_exp, e & (kExpBad - 1));
            if (e & kExpBad) s_bad = 1;
        }
    }
    __syncthreads();
    const int et = s_exp;             // |psi| < 2^(et - 1022)
    const unsigned lo = (unsigned)(et - 173) << 20;
    // weighted sums (units of 2^(et - 1122) / 831600) -> -1/2 Delta_h psi: a factor of 2^-7 to 2^-6
    // and a power of two; one thread's float64 division
    if (tid == 0) {
        int ex;
        s_cf = to_ff(d2ff(ldexp(frexp(-0.5 / ((double)kW12Den * D.h * D.h), &ex), -6)));
        s_off = et - 1122 + ex + 6;
    }
    constexpr int kWc = (int)w12_centre3();
    constexpr int kW[kHalf + 1] = {kWc,           (int)w12_int(1), (int)w12_int(2), (int)w12_int(3),
                                   (int)w12_int(4), (int)w12_int(5), (int)w12_int(6)};
    const double* const vb = v ? v + (per_system ? B.soff : B.voff) : nullptr;   // the block's potential

    const long long sy = nx, sz = (long long)nx * ny;
    IxStage sg;
    sg.init(D, P, nx, tid);
    const bool vec = (nx & 1) == 0 && (P.base & 1) == 0 && aligned16(psi);
    const int nzt = P.z1 - P.z0;
    auto copy = [&](int k, int slot) {   // plane z0 + k
        int z = P.z0 + k;
        if (per & 4) z = wrap_coord(z, nz);
        const bool okz = z < nz;
        const double* pl = psi + P.base + (okz ? z * sz : 0);
        HPair* const to = ring + slot * kIxPairs + tid;
        if (vec) {   // (one branch for the plane)
#pragma unroll
            for (int j = 0; j < kIxU; ++j)
                if (sg.wants(j, k < nzt)) sg.copy_pair(j, to + j * 256, pl, okz);
        } else {
#pragma unroll
            for (int j = 0; j < kIxU; ++j)
                if (sg.wants(j, k < nzt)) sg.copy(j, to + j * 256, pl, okz, false, nx);
        }
    };
    auto split = [&](int k, int slot) {
#pragma unroll
        for (int j = 0; j < kIxU; ++j)
            if (sg.wants(j, k < nzt)) {
                const int at = slot * kIxPairs + tid + j * 256;
                ring[at] = top_split(*reinterpret_cast<const double2*>(ring + at), lo, tops[at]);
            }
    };
    for (int k = 0; k < kHalf; ++k) copy(k, k);
    cp_async_commit();
    copy(kHalf, kHalf);
    cp_async_commit();

    const int tx = threadIdx.x, ty = threadIdx.y;     // 16 x 16; points (x0 + 2 tx + a, y0 + ty)
    const int gx = P.x0 + 2 * tx, gy = P.y0 + ty;
    const bool in0 = gx < nx && gy < ny, in1 = gx + 1 < nx && gy < ny;
    const bool ovec = (nx & 1) == 0 && (P.base & 1) == 0 && aligned16(hpsi), vvec = vec && aligned16(vb);
    const long long col = gy * sy + gx;
    const int ctr = (ty + kHalf) * (kPX / 2) + tx + kHalf / 2;   // the points' pair in a staged plane
    HPair q[kHalf];          // planes z - 6 .. z - 1
    unsigned qt[kHalf];
#pragma unroll
    for (int j = 0; j < kHalf; ++j) {   // planes z0 - 6 .. z0 - 1 straight from memory
        int z = P.z0 - kHalf + j;
        if (per & 4) z = wrap_coord(z, nz);
        const double* pl = psi + P.base + z * sz + col;
        const bool okz = z >= 0 && z < nz;
        q[j] = top_split(make_double2(okz && in0 ? pl[0] : 0.0, okz && in1 ? pl[1] : 0.0), lo, qt[j]);
    }
    asm volatile("cp.async.wait_group 1;" ::: "memory");
    for (int k = 0; k < kHalf; ++k) split(k, k);
    __syncthreads();
    const ff cf = s_cf;
    const int off = s_off;
    int slot = 0;   // of plane z0 + k
    for (int k = 0; k < nzt; ++k) {
        // the slot of plane k + 7 held plane k - 2, which every thread has finished
        if (k + 1 < nzt) copy(k + kHalf + 1, ix_slot<kHRing>(slot, kHalf + 1));
        cp_async_commit();
        asm volatile("cp.async.wait_group 1;" ::: "memory");
        const int hslot = ix_slot<kHRing>(slot, kHalf);
        split(k + kHalf, hslot);
        // psi and the potential at the plane this step computes
        double2 uc = make_double2(0.0, 0.0), vc = uc;
        const long long pz = (P.z0 + k) * sz + col;
        if (vb) {
            if (vvec) {
                if (in0) {
                    uc = *reinterpret_cast<const double2*>(psi + P.base + pz);
                    vc = *reinterpret_cast<const double2*>(vb + pz);
                }
            } else {
                if (in0) { uc.x = psi[P.base + pz]; vc.x = vb[pz]; }
                if (in1) { uc.y = psi[P.base + pz + 1]; vc.y = vb[pz + 1]; }
            }
        }
        __syncthreads();   // plane k + 6 is split, every thread has finished plane k - 1
        const HPair* const pc = ring + slot * kIxPairs + ctr;
        const unsigned* const tc = tops + slot * kIxPairs + ctr;
        HPair xw[kHalf + 1];   // columns -6 .. 7 of the row
        unsigned xt[kHalf + 1];
#pragma unroll
        for (int k2 = 0; k2 < kHalf + 1; ++k2) {
            xw[k2] = pc[k2 - kHalf / 2];
            xt[k2] = tc[k2 - kHalf / 2];
        }
        auto xh = [&](int c) { return (c & 1) ? xw[c >> 1].h.y : xw[c >> 1].h.x; };
        auto xl = [&](int c) { return (c & 1) ? xw[c >> 1].l.y : xw[c >> 1].l.x; };
        auto xtop = [&](int c) { return (c & 1) ? __byte_perm(xt[c >> 1], xt[(c >> 1) + 1], 0x5432) : xt[c >> 1]; };
        // centre, then the distances: sums and products exact in (Sh, errors), the rest in Sl
        const HPair c0 = xw[kHalf / 2];
        long long I0 = (long long)kWc * (int)(xt[kHalf / 2] & 0xffffu), I1 = (long long)kWc * (int)(xt[kHalf / 2] >> 16);
        const float2 wc = make_float2((float)kWc, (float)kWc);
        float2 Sh = __fmul2_rn(wc, c0.h);
        float2 Sl = __ffma2_rn(wc, c0.l, __ffma2_rn(wc, c0.h, make_float2(-Sh.x, -Sh.y)));
#pragma unroll
        for (int m = 1; m <= kHalf; ++m) {
            // x: one lane at a time (at odd distances the neighbours are no pairs)
            float2 e0, e1, e2, e3, e4, e5, sx;
            sx.x = two_sum(xh(kHalf - m), xh(kHalf + m), e0.x);
            sx.y = two_sum(xh(kHalf + 1 - m), xh(kHalf + 1 + m), e0.y);
            const float2 lx = make_float2(xl(kHalf - m) + xl(kHalf + m), xl(kHalf + 1 - m) + xl(kHalf + 1 + m));
            const unsigned tx2 = xtop(kHalf - m) + xtop(kHalf + m);
            const HPair ya = pc[-m * (kPX / 2)], yb = pc[m * (kPX / 2)];
            const int zs = ix_slot<kHRing>(slot, m) * kIxPairs + ctr;
            const HPair za = q[kHalf - m], zb = ring[zs];
            const unsigned t = tx2 + (tc[-m * (kPX / 2)] + tc[m * (kPX / 2)]) + (qt[kHalf - m] + tops[zs]);
            I0 += (long long)kW[m] * (int)(t & 0xffffu);
            I1 += (long long)kW[m] * (int)(t >> 16);
            const float2 sy2 = two_sum2(ya.h, yb.h, e1), sz2 = two_sum2(za.h, zb.h, e2);
            const float2 s = two_sum2(two_sum2(sx, sy2, e3), sz2, e4);
            float2 l = __fadd2_rn(__fadd2_rn(lx, __fadd2_rn(ya.l, yb.l)), __fadd2_rn(za.l, zb.l));
            l = __fadd2_rn(l, __fadd2_rn(__fadd2_rn(e0, e1), __fadd2_rn(e2, __fadd2_rn(e3, e4))));
            const float2 w = make_float2((float)kW[m], (float)kW[m]);
            const float2 p = __fmul2_rn(w, s);
            const float2 ep = __ffma2_rn(w, s, make_float2(-p.x, -p.y));
            Sh = two_sum2(Sh, p, e5);
            Sl = __fadd2_rn(__ffma2_rn(w, l, Sl), __fadd2_rn(ep, e5));
        }
        slot = ix_slot<kHRing>(slot, 1);
        double r[2];
        top_join(I0, I1, Sh, Sl, cf, off, r);
        if (vb) {
            r[0] = fma(vc.x, uc.x, r[0]);
            r[1] = fma(vc.y, uc.y, r[1]);
        }
        double* const o = hpsi + P.base + pz;
        if (ovec) {
            if (in0) *reinterpret_cast<double2*>(o) = make_double2(r[0], r[1]);
        } else {
            if (in0) o[0] = r[0];
            if (in1) o[1] = r[1];
        }
#pragma unroll
        for (int j = 0; j + 1 < kHalf; ++j) {
            q[j] = q[j + 1];
            qt[j] = qt[j + 1];
        }
        q[kHalf - 1] = c0;
        qt[kHalf - 1] = xt[kHalf / 2];
    }
    if (s_bad) {   // NaN wherever a tap reads a value out of range (the float-float sweep did so too)
        for (int z = P.z0; z < P.z1; ++z)
            for (int a = 0; a < 2; ++a) {
                if (!(a == 0 ? in0 : in1)) continue;
                bool fin = true;
                for (int d = 0; d < 3; ++d)
                    for (int m = -kHalf; m <= kHalf; ++m) {
                        int px = gx + a + (d == 0 ? m : 0), py = gy + (d == 1 ? m : 0), zz = z + (d == 2 ? m : 0);
                        if (per & 1) px = wrap_coord(px, nx);
                        if (per & 2) py = wrap_coord(py, ny);
                        if (per & 4) zz = wrap_coord(zz, nz);
                        if (px < 0 || px >= nx || py < 0 || py >= ny || zz < 0 || zz >= nz) continue;
                        fin = fin && expo(psi[P.base + zz * sz + py * sy + px]) <= kExpMax;
                    }
                if (!fin) hpsi[P.base + z * sz + col + a] = __longlong_as_double(0x7ff8000000000000LL);
            }
    }
}

// float64: plain loads of the 37 taps (through L1), float64 arithmetic.
__global__ void __launch_bounds__(256) k_hamiltonian64(const BlkDesc* __restrict__ blk, const LvlDesc* __restrict__ L,
                                                       const int4* __restrict__ tiles, const int* __restrict__ orb_blk,
                                                       const double* __restrict__ psi, const double* __restrict__ vloc,
                                                       const double* __restrict__ vavg, double* __restrict__ hpsi) {
    const TilePos P = tile_pos(blk, L, tiles, orb_blk, blockIdx.x);
    const LvlDesc& D = L[P.b];
    const BlkDesc& B = blk[P.b];
    double w[kHalf + 1];
#pragma unroll
    for (int m = 0; m <= kHalf; ++m) w[m] = c_w64[m];
    const double mh = -0.5 / (D.h * D.h);
    const long long sy = D.nx, sz = (long long)D.nx * D.ny;
    const int x = P.x0 + threadIdx.x;
    if (x >= D.nx) return;
    for (int k = 0; k < 2; ++k) {
        const int y = P.y0 + threadIdx.y + k * (kTileY / 2);
        if (y >= D.ny) continue;
        for (int z = P.z0; z < P.z1; ++z) {
            const long long q = (long long)z * sz + y * sy + x;
            const long long g = P.base + q;
            const double u = psi[g];
            double acc = 3.0 * w[0] * u;
            for (int m = 1; m <= kHalf; ++m) {
                double s = 0.0;
                if (x - m >= 0) s += psi[g - m];
                if (x + m < D.nx) s += psi[g + m];
                if (y - m >= 0) s += psi[g - m * sy];
                if (y + m < D.ny) s += psi[g + m * sy];
                if (z - m >= 0) s += psi[g - m * sz];
                if (z + m < D.nz) s += psi[g + m * sz];
                acc += w[m] * s;
            }
            double v = 0.0;
            if (vloc) v += vloc[B.soff + q];
            if (vavg) v += vavg[B.voff + q];
            hpsi[g] = mh * acc + v * u;
        }
    }
}

void launch_hamiltonian(const flosic_ctx* c, const double* psi, const double* vloc, const double* vavg,
                        double* hpsi, cudaStream_t s) {
    const Multigrid& M = c->mg;
    const dim3 tb(kTileX, kTileY / 2);
    if (c->opt.precision == FLOSIC_MIXED) {
        k_tile_exp<<<(unsigned)M.ntiles[0], tb, 0, s>>>(c->d_blk, M.d_lvl[0], M.d_tiles[0], c->d_orb_blk, psi, vloc, vavg,
                                                        c->ws.vsum, c->ws.texp);
        note_launch((flosic_ctx*)c);
        const double* v = vloc && vavg ? c->ws.vsum : (vloc ? vloc : vavg);
        k_hamiltonian_mixed<<<(unsigned)M.ntiles[0], dim3(kTileX / 2, kTileY), kHSmem, s>>>(
            c->d_blk, M.d_lvl[0], M.d_tiles[0], c->d_orb_blk, psi, v, vloc && !vavg ? 1 : 0, c->ws.texp, hpsi);
    } else
        k_hamiltonian64<<<(unsigned)M.ntiles[0], tb, 0, s>>>(c->d_blk, M.d_lvl[0], M.d_tiles[0], c->d_orb_blk, psi,
                                                              vloc, vavg, hpsi);
    note_launch((flosic_ctx*)c);
}

cudaError_t upload_hamiltonian_constants() {
    double w[kHalf + 1];
    stencil_weights(w);
    const cudaError_t e = cudaMemcpyToSymbol(c_w64, w, sizeof(w));
    if (e != cudaSuccess) return e;
    return ensure_dyn_smem((const void*)k_hamiltonian_mixed, kHSmem);
}

}  // namespace flosic
