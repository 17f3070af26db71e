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
// Mixed precision: the Laplacian in exact integer sums (ixsweep.cuh).
//
// A tile's psi (with the halo its taps reach) lies below 2^k, k from the
// tiles' largest exponents (k_tile_exp).  Every staged value becomes the
// integer q = trunc(psi 2^(57-k)) in two digits, q = hi 2^29 + lo with
// |hi|, |lo| <= 2^28; both digit fields are summed and weighted in integers,
// so the only rounding of the Laplacian is the 2^-57 of the tile's largest
// value (the float-float sweep that this replaced held 2^-48 of each value) and
// the final float64 result, which takes three float64 operations per point.
//
// What bounds it: instruction issue and the latencies of 16 warps per SM (310
// instructions per point, 46 % of the issue slots; 128 registers a thread hold
// the z-windows).  The two digits need 6 integer additions (three-operand) and
// 2 multiply-adds per distance, against error-free sums and products of pairs.
// A value is split once, when its plane arrives (IxStage); one barrier per
// plane.  With the z-loop unrolled 13 times, which keeps every window slot in
// place, a third of the issue slots waited for instructions (2.7 -> 3.5 ms).
// 128^3 x 64 orbitals with both potentials: 5.82 -> 2.24 ms, of which
// k_tile_exp 0.15.
// ---------------------------------------------------------------------------
constexpr int kHSmem = kIxPts * 8 * kIxRing;
constexpr int kExpBad = 1 << 16;                     // a tile with a value beyond 2^799, an infinity or a NaN
constexpr int kExpMin = 223, kExpMax = 1821;         // biased exponents in use: the scales stay normal float64
                                                     // (smaller psi count as zero)
__device__ __forceinline__ int expo(double v) { return (__double2hiint(v) >> 20) & 0x7ff; }

// Per tile: the largest biased exponent of its psi, + kExpBad.
__global__ void __launch_bounds__(256) k_tile_exp(const BlkDesc* __restrict__ blk, const LvlDesc* __restrict__ L,
                                                  const int4* __restrict__ tiles, const int* __restrict__ orb_blk,
                                                  const double* __restrict__ psi, int* __restrict__ texp) {
    __shared__ int s_max, s_bad;
    const TilePos P = tile_pos(blk, L, tiles, orb_blk, blockIdx.x);
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

// trunc(v 2^(1079 - et)) as digits (hi, lo); et at least kExpMin and at least
// v's biased exponent (what lies above it becomes 0: the staged corners, which
// no tap reads, and the values that make a tile bad).
__device__ __forceinline__ int2 ix_digits(double v, int et) {
    const int hw = __double2hiint(v);
    const unsigned sh = min((unsigned)(et - ((hw >> 20) & 0x7ff)), 63u);
    const unsigned long long m =
        ((unsigned long long)(unsigned)((hw & 0xfffff) | 0x100000) << 32) | (unsigned)__double2loint(v);
    const long long sg = hw >> 31;
    const long long q = ((long long)((m << 4) >> sh) ^ sg) - sg;
    const long long t = q + (1 << 28);
    return make_int2((int)(t >> 29), (int)((unsigned)t & 0x1fffffffu) - (1 << 28));
}

// H 2^10 + L 2^-19 (H, L weighted sums of hi and lo digits, below 2^53 in
// magnitude) in float64, built with integer operations: the sum as an integer
// (2^-10 of a unit of H, a quarter of the digits' own resolution after
// weighting), normalised and truncated to 53 bits.
__device__ __forceinline__ double ix_to_double(long long H, long long L) {
    const long long t = (H << 10) + ((L + (1 << 18)) >> 19);
    const long long sg = t >> 63;
    const unsigned long long a = (unsigned long long)((t ^ sg) - sg);
    if (a == 0) return 0.0;
    const int lz = __clzll((long long)a);
    const unsigned long long m = a << lz;   // its top bit adds 1 to the exponent
    const unsigned hw = ((unsigned)(1023 + 62 - lz) << 20) + (unsigned)(m >> 43);
    return __hiloint2double((int)(hw | ((unsigned)sg & 0x80000000u)), (int)(unsigned)(m >> 11));
}

__global__ void __launch_bounds__(256, 2) k_hamiltonian_ix(const BlkDesc* __restrict__ blk, const LvlDesc* __restrict__ L,
                                                           const int4* __restrict__ tiles,
                                                           const int* __restrict__ orb_blk,
                                                           const double* __restrict__ psi,
                                                           const double* __restrict__ vloc,
                                                           const double* __restrict__ vavg,
                                                           const int* __restrict__ texp, double* __restrict__ hpsi) {
    extern __shared__ __align__(16) unsigned char hs_raw[];
    int2* const ring = reinterpret_cast<int2*>(hs_raw);
    __shared__ int s_exp, s_bad;
    __shared__ double s_cf;
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
    {   // the largest exponent among this tile and those its taps reach (periodic: the orbital's)
        const int ntx = (nx + kTileX - 1) / kTileX, nty = (ny + kTileY - 1) / kTileY;
        int e = 0, bad = 0;   // (apart: a flag in e would outweigh every later exponent)
        auto take = [&](int v) {
            e = max(e, v & (kExpBad - 1));
            bad |= v & kExpBad;
        };
        if (per) {
            for (int t = tid; t < D.ntile; t += 256) take(texp[P.first + t]);
        } else if (tid < 32) {
            const int kx = P.x0 / kTileX, ky = P.y0 / kTileY;
            const int kz0 = max(P.z0 - kHalf, 0) / D.tz, kz1 = min(P.z1 + kHalf - 1, nz - 1) / D.tz;
            int jx = kx, jy = ky, jz = kz0 + tid - 4;   // lanes 4 ..: the column's tiles
            bool ok = tid >= 4 && jz <= kz1;
            if (tid < 4) {
                jz = P.z0 / D.tz;
                if (tid < 2) jx += 2 * tid - 1;
                else jy += 2 * tid - 5;
                ok = jx >= 0 && jx < ntx && jy >= 0 && jy < nty;
            }
            if (ok) take(texp[P.first + ((long long)jz * nty + jy) * ntx + jx]);
        }
        if (e) atomicMax(&s_exp, e);
        if (bad) s_bad = 1;
        __syncthreads();
    }
    const int et = s_exp;             // |psi| < 2^(et - 1022)
    // weighted sums (units of 2^(et - 1022 - 38) / 831600) -> -h^2/2 Delta_h psi; one thread's float64 division
    if (tid == 0) s_cf = scalbn(-0.5 / ((double)kW12Den * D.h * D.h), et - 1022 - 38);
    constexpr int kWc = (int)w12_centre3();
    constexpr int kW[kHalf + 1] = {kWc,           (int)w12_int(1), (int)w12_int(2), (int)w12_int(3),
                                   (int)w12_int(4), (int)w12_int(5), (int)w12_int(6)};
    const bool pot = vloc != nullptr || vavg != nullptr;

    const long long sy = nx, sz = (long long)nx * ny;
    IxStage sg;
    sg.init(D, P, nx, tid);
    const bool vec = (nx & 1) == 0 && (P.base & 1) == 0 && ((reinterpret_cast<uintptr_t>(psi) & 15) == 0);
    const int nzt = P.z1 - P.z0;
    auto copy = [&](int k, int slot) {   // plane z0 + k
        int z = P.z0 + k;
        if (per & 4) z = wrap_coord(z, nz);
        const bool okz = z < nz;
        const double* pl = psi + P.base + (okz ? z * sz : 0);
#pragma unroll
        for (int j = 0; j < kIxU; ++j)
            if (sg.wants(j, k < nzt)) sg.copy(j, ring + slot * kIxPts + 2 * (tid + j * 256), pl, okz, vec, nx);
    };
    auto split = [&](int k, int slot) {
#pragma unroll
        for (int j = 0; j < kIxU; ++j)
            if (sg.wants(j, k < nzt)) {
                int2* const at = ring + slot * kIxPts + 2 * (tid + j * 256);
                const double2 v = *reinterpret_cast<const double2*>(at);
                const int2 d0 = ix_digits(v.x, et), d1 = ix_digits(v.y, et);
                *reinterpret_cast<int4*>(at) = make_int4(d0.x, d0.y, d1.x, d1.y);
            }
    };
    for (int k = 0; k < kHalf; ++k) copy(k, k);
    cp_async_commit();
    copy(kHalf, kHalf);
    cp_async_commit();
    copy(kHalf + 1, kHalf + 1);
    cp_async_commit();

    const int tx = threadIdx.x, ty = threadIdx.y;     // 16 x 16; points (x0 + 2 tx + a, y0 + ty)
    const int gx = P.x0 + 2 * tx, gy = P.y0 + ty;
    const bool in0 = gx < nx && gy < ny, in1 = gx + 1 < nx && gy < ny;
    const bool ovec = (nx & 1) == 0 && (P.base & 1) == 0 && ((reinterpret_cast<uintptr_t>(hpsi) & 15) == 0);
    const long long col = gy * sy + gx;
    const int ctr = (ty + kHalf) * kPX + 2 * tx + kHalf;   // the first point in a staged plane
    int2 q0[kQ], q1[kQ];   // z-windows: step k0 + u's in slots u .. u + 12
#pragma unroll
    for (int j = 0; j < kHalf; ++j) {   // planes z0 - 6 .. z0 - 1 straight from memory
        int z = P.z0 - kHalf + j;
        if (per & 4) z = wrap_coord(z, nz);
        const double* pl = psi + P.base + z * sz + col;
        q0[j] = ix_digits(z >= 0 && z < nz && in0 ? pl[0] : 0.0, et);
        q1[j] = ix_digits(z >= 0 && z < nz && in1 ? pl[1] : 0.0, et);
    }
    asm volatile("cp.async.wait_group 2;" ::: "memory");
    for (int k = 0; k < kHalf; ++k) split(k, k);
    __syncthreads();
    const double cf = s_cf;
#pragma unroll
    for (int k = 0; k < kHalf; ++k) {
        const int4 hv = *reinterpret_cast<const int4*>(ring + k * kIxPts + ctr);
        q0[kHalf + k] = make_int2(hv.x, hv.y);
        q1[kHalf + k] = make_int2(hv.z, hv.w);
    }
    int slot = 0;   // of plane z0 + k
    for (int k0 = 0; k0 < nzt; k0 += kZU) {
#pragma unroll
        for (int u = 0; u < kZU; ++u) {
            const int k = k0 + u;
            if (k >= nzt) break;
            // the slot of plane k + 8 held plane k - 2, which every thread has finished
            if (k + 2 < nzt) copy(k + kHalf + 2, ix_slot(slot, kHalf + 2));
            cp_async_commit();
            asm volatile("cp.async.wait_group 2;" ::: "memory");
            const int hslot = ix_slot(slot, kHalf);
            split(k + kHalf, hslot);
            // psi and the potential at the plane this step computes
            double uc[2] = {0.0, 0.0}, va[2] = {0.0, 0.0}, vb[2] = {0.0, 0.0};
            const long long pz = (P.z0 + k) * sz + col;
            if (pot) {
#pragma unroll
                for (int a = 0; a < 2; ++a)
                    if (a == 0 ? in0 : in1) {
                        uc[a] = psi[P.base + pz + a];
                        if (vloc) va[a] = vloc[B.soff + pz + a];
                        if (vavg) vb[a] = vavg[B.voff + pz + a];
                    }
            }
            __syncthreads();   // plane k + 6 is split, every thread has finished plane k - 1
            {
                const int4 hv = *reinterpret_cast<const int4*>(ring + hslot * kIxPts + ctr);
                q0[u + 2 * kHalf] = make_int2(hv.x, hv.y);
                q1[u + 2 * kHalf] = make_int2(hv.z, hv.w);
            }
            const int2* const pc = ring + slot * kIxPts + ctr;
            slot = ix_slot(slot, 1);
            int2 xw[2 * kHalf + 2];   // columns -6 .. 7 of the row
#pragma unroll
            for (int k2 = 0; k2 < kHalf + 1; ++k2) {
                const int4 v = *reinterpret_cast<const int4*>(pc - kHalf + 2 * k2);
                xw[2 * k2] = make_int2(v.x, v.y);
                xw[2 * k2 + 1] = make_int2(v.z, v.w);
            }
            const int2 c0 = q0[u + kHalf], c1 = q1[u + kHalf];
            long long H0 = (long long)kWc * c0.x, L0 = (long long)kWc * c0.y;
            long long H1 = (long long)kWc * c1.x, L1 = (long long)kWc * c1.y;
#pragma unroll
            for (int m = 1; m <= kHalf; ++m) {
                const int4 uu = *reinterpret_cast<const int4*>(pc - m * kPX);
                const int4 ww = *reinterpret_cast<const int4*>(pc + m * kPX);
                const int2 a0 = q0[u + kHalf - m], b0 = q0[u + kHalf + m];
                const int2 a1 = q1[u + kHalf - m], b1 = q1[u + kHalf + m];
                H0 += (long long)kW[m] * (xw[kHalf - m].x + xw[kHalf + m].x + uu.x + ww.x + a0.x + b0.x);
                L0 += (long long)kW[m] * (xw[kHalf - m].y + xw[kHalf + m].y + uu.y + ww.y + a0.y + b0.y);
                H1 += (long long)kW[m] * (xw[kHalf + 1 - m].x + xw[kHalf + 1 + m].x + uu.z + ww.z + a1.x + b1.x);
                L1 += (long long)kW[m] * (xw[kHalf + 1 - m].y + xw[kHalf + 1 + m].y + uu.w + ww.w + a1.y + b1.y);
            }
            double r[2] = {ix_to_double(H0, L0) * cf, ix_to_double(H1, L1) * cf};
            if (pot) {
#pragma unroll
                for (int a = 0; a < 2; ++a) r[a] = fma(vloc && vavg ? va[a] + vb[a] : (vloc ? va[a] : vb[a]), uc[a], r[a]);
            }
            double* const o = hpsi + P.base + pz;
            if (ovec) {
                if (in0) *reinterpret_cast<double2*>(o) = make_double2(r[0], r[1]);
            } else {
                if (in0) o[0] = r[0];
                if (in1) o[1] = r[1];
            }
        }
        ix_shift(q0);
        ix_shift(q1);
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
        k_tile_exp<<<(unsigned)M.ntiles[0], tb, 0, s>>>(c->d_blk, M.d_lvl[0], M.d_tiles[0], c->d_orb_blk, psi,
                                                                 c->ws.texp);
        note_launch((flosic_ctx*)c);
        k_hamiltonian_ix<<<(unsigned)M.ntiles[0], dim3(kTileX / 2, kTileY), kHSmem, s>>>(
            c->d_blk, M.d_lvl[0], M.d_tiles[0], c->d_orb_blk, psi, vloc, vavg, c->ws.texp, hpsi);
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
    return ensure_dyn_smem((const void*)k_hamiltonian_ix, kHSmem);
}

}  // namespace flosic
