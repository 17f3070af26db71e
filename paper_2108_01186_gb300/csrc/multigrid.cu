// Multigrid preconditioner of the Poisson CG (Sec. II.A solves the
// electrostatics iteratively; the solver here is preconditioned CG).
//
// M ~ A2^{-1}, one V-cycle on the 7-point Laplacian A2 (spacing 2^l h on
// level l, zero outside the interior).  A2 and the 12th-order operator A
// satisfy 1 <= x^T A x / x^T A2 x <= 1.77 for every grid function vanishing
// outside the interior (the ratio of their Fourier symbols), so CG on A with
// this preconditioner converges in a few tens of iterations at any grid
// size instead of O(n).
//
// Vertex-centred coarsening: coarse point I sits on fine point 2I+1,
// n_c = floor(n/2); coarsen while every side is >= 6.  On an even side the
// last coarse point is the last fine point, so the coarse grid's zero
// boundary would sit one coarse spacing out while the true one is closer:
// the 7-point operator of such a level keeps the off-diagonal -1/h_l^2 but
// takes at the last point of that dimension the diagonal weight of the 1-D
// Galerkin operator P^T A P / 2 (c' = 2c - 1 for an even parent side,
// 1 + c/2 for an odd one, c = 2 on the fine grid).  Without it the V-cycle
// loses most of its strength on grids such as 128^3.  Restriction is full
// weighting (1/4, 1/2, 1/4 per direction) = (1/8) P^T with P trilinear
// interpolation.  Smoother: one damped-Jacobi sweep before and after
// (omega = 0.8); coarsest level: 40 damped-Jacobi sweeps from zero.  Every
// piece is symmetric and the smoother converges in the A2 norm, so the V-cycle
// is a symmetric positive definite operator.
//
// Kernels work on per-level tables of 3-D tiles (one CTA of 32 x 8 threads per
// 32 x 16 column of one orbital, as many planes deep as tile_depth and
// tile_split say; neighbours come through L1) so that all orbitals of all systems run in one launch
// per level; the levels small enough for shared memory run in one launch
// together (k_mg_coarse).
#include "internal.cuh"

namespace flosic {

// sum of the six neighbours (zero outside)
template <class T>
__device__ __forceinline__ T nbr6(const T* __restrict__ u, long long g, int x, int y, int z, const LvlDesc& D) {
    const long long sy = D.nx, sz = (long long)D.nx * D.ny;
    T s = 0;
    if (x > 0) s += u[g - 1];
    if (x < D.nx - 1) s += u[g + 1];
    if (y > 0) s += u[g - sy];
    if (y < D.ny - 1) s += u[g + sy];
    if (z > 0) s += u[g - sz];
    if (z < D.nz - 1) s += u[g + sz];
    return s;
}

// 1 / (sum of the diagonal weights) at (x, y, z) of a level: 1/6 away from
// the last point of every dimension.
template <class T>
__device__ __forceinline__ T inv_diag(const LvlDesc& D, int x, int y, int z) {
    const int m = (x == D.nx - 1 ? 1 : 0) | (y == D.ny - 1 ? 2 : 0) | (z == D.nz - 1 ? 4 : 0);
    return T(D.idd[m]);
}

template <class T> struct Vec2;
template <> struct Vec2<float> { using type = float2; };
template <> struct Vec2<double> { using type = double2; };

// Gathers, for n consecutive points starting at (x, y, z) (n = vector width
// or 1), the centre values and the sum of the six neighbours (zero outside).
template <class T, int V>
__device__ __forceinline__ void centre_nbr(const T* __restrict__ u, const LvlDesc& D, int x, int y, int z,
                                           long long g, int n, T* c, T* nb) {
    using VT = typename Vec<T>::type;
    const long long sy = D.nx, sz = (long long)D.nx * D.ny;
    if (n == V) {
        const VT cv = *reinterpret_cast<const VT*>(u + g);
        VT ym, yp, zm, zp;
        const T* cs = reinterpret_cast<const T*>(&cv);
        T zero[V];
#pragma unroll
        for (int k = 0; k < V; ++k) zero[k] = T(0);
        ym = (y > 0) ? *reinterpret_cast<const VT*>(u + g - sy) : *reinterpret_cast<const VT*>(zero);
        yp = (y < D.ny - 1) ? *reinterpret_cast<const VT*>(u + g + sy) : *reinterpret_cast<const VT*>(zero);
        zm = (z > 0) ? *reinterpret_cast<const VT*>(u + g - sz) : *reinterpret_cast<const VT*>(zero);
        zp = (z < D.nz - 1) ? *reinterpret_cast<const VT*>(u + g + sz) : *reinterpret_cast<const VT*>(zero);
        const T xl = (x > 0) ? u[g - 1] : T(0);
        const T xr = (x + V < D.nx) ? u[g + V] : T(0);
        const T* a = reinterpret_cast<const T*>(&ym);
        const T* b = reinterpret_cast<const T*>(&yp);
        const T* cz = reinterpret_cast<const T*>(&zm);
        const T* d = reinterpret_cast<const T*>(&zp);
#pragma unroll
        for (int k = 0; k < V; ++k) {
            c[k] = cs[k];
            const T left = (k == 0) ? xl : cs[k - 1];
            const T right = (k == V - 1) ? xr : cs[k + 1];
            nb[k] = left + right + a[k] + b[k] + cz[k] + d[k];
        }
    } else {
        c[0] = u[g];
        T sum = 0;
        if (x > 0) sum += u[g - 1];
        if (x < D.nx - 1) sum += u[g + 1];
        if (y > 0) sum += u[g - sy];
        if (y < D.ny - 1) sum += u[g + sy];
        if (z > 0) sum += u[g - sz];
        if (z < D.nz - 1) sum += u[g + sz];
        nb[0] = sum;
    }
}

template <class T, int V>
__device__ __forceinline__ void store_n(T* dst, const T* v, int n) {
    using VT = typename Vec<T>::type;
    if (n == V) *reinterpret_cast<VT*>(dst) = *reinterpret_cast<const VT*>(v);
    else dst[0] = v[0];
}

// s = r - A2 (omega D^-1 r) = (1 - omega) r + omega sum_nbr r / dd(nbr),
// dd = 6 except on the last points of a level with corrected weights.
template <class T>
__global__ void __launch_bounds__(256) k_mg_resid_smooth(const BlkDesc* __restrict__ blk, const LvlDesc* __restrict__ L,
                                                         const int4* __restrict__ tiles, const int* __restrict__ orb_blk,
                                                         const int* __restrict__ active, const T* __restrict__ r,
                                                         T* __restrict__ s, T omega) {
    constexpr int V = Vec<T>::n;
    const TilePos P = tile_pos(blk, L, tiles, orb_blk, blockIdx.x);
    const LvlDesc& D = L[P.b];
    if (!active[P.o] || D.fused) return;
    const long long sy = D.nx, sz = (long long)D.nx * D.ny;
    tile_rows<T>(D, P, [&](int x, int y, int z, long long g, int n) {
        if (D.corr && (x + n >= D.nx - 1 || y >= D.ny - 2 || z >= D.nz - 2)) {
            // a neighbour may lie on a last point: weight each one
            for (int k = 0; k < n; ++k) {
                const int xk = x + k;
                const long long gk = g + k;
                T sum = T(0);
                if (xk > 0) sum += r[gk - 1] * inv_diag<T>(D, xk - 1, y, z);
                if (xk < D.nx - 1) sum += r[gk + 1] * inv_diag<T>(D, xk + 1, y, z);
                if (y > 0) sum += r[gk - sy] * inv_diag<T>(D, xk, y - 1, z);
                if (y < D.ny - 1) sum += r[gk + sy] * inv_diag<T>(D, xk, y + 1, z);
                if (z > 0) sum += r[gk - sz] * inv_diag<T>(D, xk, y, z - 1);
                if (z < D.nz - 1) sum += r[gk + sz] * inv_diag<T>(D, xk, y, z + 1);
                s[gk] = (T(1) - omega) * r[gk] + omega * sum;
            }
            return;
        }
        T c[V], nb[V], out[V];
        centre_nbr<T, V>(r, D, x, y, z, g, n, c, nb);
#pragma unroll
        for (int k = 0; k < V; ++k) out[k] = (T(1) - omega) * c[k] + omega * T(1.0 / 6.0) * nb[k];
        store_n<T, V>(s + g, out, n);
    });
}

// r_c(I) = sum over the 27 fine neighbours of 2I+1 of (1/4,1/2,1/4)^3 s_f;
// V consecutive coarse points per thread, fine rows read with vector loads
// when they are aligned.
template <class T>
__global__ void __launch_bounds__(256) k_mg_restrict(const BlkDesc* __restrict__ blk, const LvlDesc* __restrict__ Lc,
                                                     const LvlDesc* __restrict__ Lf, const int4* __restrict__ tiles_c,
                                                     const int* __restrict__ orb_blk, const int* __restrict__ active,
                                                     const T* __restrict__ sf, T* __restrict__ rc) {
    constexpr int V = Vec<T>::n;
    using VT = typename Vec<T>::type;
    const TilePos P = tile_pos(blk, Lc, tiles_c, orb_blk, blockIdx.x);
    const LvlDesc& C = Lc[P.b];
    const LvlDesc& F = Lf[P.b];
    if (!active[P.o] || F.fused) return;
    const long long fbase = F.off + (long long)(P.o - blk[P.b].orb0) * F.G;
    const T* fb = sf + fbase;
    const long long fy = F.nx, fz = (long long)F.nx * F.ny;
    const bool fvec = (F.nx % (2 * V) == 0) && (fbase % (2 * V) == 0);
    // float64: the nine fine rows' loads in flight together (48^3 x 40 89 against 97 us,
    // 64^3 x 6 19.6 and 21.0).  float32 takes the rows one after the other: nine at once
    // cost registers (128^3 x 24 68 against 56 us, 117^3 x 16 124 and 72, 64^3 x 10 8.2
    // and 6.1, 33^3 x 5 7.7 and 5.9)
    constexpr bool kAhead = sizeof(T) == sizeof(double);
    constexpr int kU = kAhead ? 3 : 1;
    tile_rows<T>(C, P, [&](int X, int Y, int Z, long long g, int n) {
        T acc[V];
#pragma unroll
        for (int k = 0; k < V; ++k) acc[k] = T(0);
        const int xf0 = 2 * X;
#pragma unroll kU
        for (int c = 0; c < 3; ++c) {
            const int zf = 2 * Z + c;
            const T wc = (c == 1) ? T(0.5) : T(0.25);
#pragma unroll kU
            for (int b = 0; b < 3; ++b) {
                const int yf = 2 * Y + b;
                const bool ok = zf < F.nz && yf < F.ny;   // rows past the grid count as zero
                if (!kAhead && !ok) continue;
                const T w = wc * ((b == 1) ? T(0.5) : T(0.25));
                const T* row = fb + (ok ? zf * fz + yf * fy : 0);
                T f[2 * V + 1];
                if (n == V && fvec) {
                    VT a0{}, a1{};
                    if (ok) {
                        a0 = *reinterpret_cast<const VT*>(row + xf0);
                        a1 = *reinterpret_cast<const VT*>(row + xf0 + V);
                    }
#pragma unroll
                    for (int k = 0; k < V; ++k) {
                        f[k] = reinterpret_cast<const T*>(&a0)[k];
                        f[V + k] = reinterpret_cast<const T*>(&a1)[k];
                    }
                    f[2 * V] = (ok && xf0 + 2 * V < F.nx) ? row[xf0 + 2 * V] : T(0);
                } else {
#pragma unroll
                    for (int k = 0; k < 2 * V + 1; ++k) f[k] = (ok && xf0 + k < F.nx) ? row[xf0 + k] : T(0);
                }
#pragma unroll
                for (int k = 0; k < V; ++k)
                    acc[k] += w * (T(0.25) * f[2 * k] + T(0.5) * f[2 * k + 1] + T(0.25) * f[2 * k + 2]);
            }
        }
        store_n<T, V>(rc + g, acc, n);
    });
}

// trilinear prolongation at fine x from one coarse row (OOB zero)
template <class T>
__device__ __forceinline__ T prolong_x(const T* __restrict__ row, int ncx, int x) {
    if (x & 1) {
        const int I = (x - 1) >> 1;
        return (I < ncx) ? row[I] : T(0);
    }
    const int I0 = (x >> 1) - 1, I1 = x >> 1;
    T v = 0;
    if (I0 >= 0) v += row[I0];
    if (I1 < ncx) v += row[I1];
    return T(0.5) * v;
}

// Coarse rows of a fine row along y (or z): odd y sits on coarse (y-1)/2,
// even y halfway between y/2-1 and y/2 (rows outside the coarse grid drop).
template <class T>
__device__ __forceinline__ int coarse_rows(int y, int nc, int* J, T* w) {
    if (y & 1) {
        J[0] = (y - 1) >> 1;
        w[0] = T(1);
        return 1;
    }
    const int lo = (y >> 1) - 1, hi = y >> 1;
    const bool vlo = lo >= 0, vhi = hi < nc;
    J[0] = vlo ? lo : hi;
    J[1] = hi;
    w[0] = w[1] = T(0.5);
    return (vlo && vhi) ? 2 : 1;
}

// t = omega D^-1 r + P e_c (pre-smoothed part plus the coarse correction)
// for the V consecutive fine points (x .. x+n-1) of one row: their trilinear
// values come from the 1, 2 or 4 coarse rows around the row.
template <class T>
__device__ __forceinline__ void prolong_row(const LvlDesc& F, const LvlDesc& C, const T* __restrict__ eb,
                                            const T* __restrict__ r, T* __restrict__ t, T oh2, int x, int y, int z,
                                            long long g, int n) {
    constexpr int V = Vec<T>::n;
    using VT = typename Vec<T>::type;
    int Jr[2], Kr[2];
    T wy[2], wz[2];
    const int nj = coarse_rows<T>(y, C.ny, Jr, wy);
    const int nk = coarse_rows<T>(z, C.nz, Kr, wz);
    T u[V];
#pragma unroll
    for (int k = 0; k < V; ++k) u[k] = T(0);
#pragma unroll
    for (int b = 0; b < 2; ++b) {
        if (b >= nk) continue;
#pragma unroll
        for (int a = 0; a < 2; ++a) {
            if (a >= nj) continue;
            const T* row = eb + ((long long)Kr[b] * C.ny + Jr[a]) * C.nx;
            const T w = wy[a] * wz[b];
            if (n == V) {
                // x is a multiple of V and F.nx of V, so C.nx = F.nx / 2
                const int I = x >> 1;
                const T e0 = (I >= 1) ? row[I - 1] : T(0);
                const T e1 = row[I];
                if (V == 4) {
                    const T e2 = row[I + 1];
                    u[0] += w * T(0.5) * (e0 + e1);
                    u[1] += w * e1;
                    u[2] += w * T(0.5) * (e1 + e2);
                    u[3] += w * e2;
                } else {
                    u[0] += w * T(0.5) * (e0 + e1);
                    u[1] += w * e1;
                }
            } else {
                u[0] += w * prolong_x(row, C.nx, x);
            }
        }
    }
    T rv[V], out[V];
    if (n == V) {
        const VT v = *reinterpret_cast<const VT*>(r + g);
#pragma unroll
        for (int k = 0; k < V; ++k) rv[k] = reinterpret_cast<const T*>(&v)[k];
    } else {
        rv[0] = r[g];
    }
    const bool edge = F.corr && (x + n >= F.nx || y == F.ny - 1 || z == F.nz - 1);
#pragma unroll
    for (int k = 0; k < V; ++k) {
        const T d = oh2 * (edge ? inv_diag<T>(F, x + k, y, z) : T(1.0 / 6.0));
        out[k] = d * rv[k] + u[k];
    }
    store_n<T, V>(t + g, out, n);
}

// Prolongation kernel.  float32 rows aligned to 4 go four rows at a time: the
// fine rows (y, y+1) x (z, z+1), y and z even, share the coarse rows J-1, J
// and K-1, K (J = y/2, K = z/2), so one thread loads those four coarse rows
// (three values each, zero outside the coarse grid) and all four fine rows
// at once.  Everything else goes row by row.
template <class T>
__global__ void __launch_bounds__(256) k_mg_prolong(const BlkDesc* __restrict__ blk, const LvlDesc* __restrict__ Lf,
                                                    const LvlDesc* __restrict__ Lc, const int4* __restrict__ tiles_f,
                                                    const int* __restrict__ orb_blk, const int* __restrict__ active,
                                                    const T* __restrict__ r, const T* __restrict__ ec,
                                                    T* __restrict__ t, T omega) {
    const TilePos P = tile_pos(blk, Lf, tiles_f, orb_blk, blockIdx.x);
    const LvlDesc& F = Lf[P.b];
    if (!active[P.o] || F.fused) return;
    const LvlDesc& C = Lc[P.b];
    const T* eb = ec + C.off + (long long)(P.o - blk[P.b].orb0) * C.G;
    const T oh2 = omega * T(F.h * F.h);
    constexpr bool kQuad = sizeof(T) == sizeof(float);
    if (!kQuad || F.corr || (F.nx % 4) != 0 || (P.base % 4) != 0) {
        tile_rows<T>(F, P, [&](int x, int y, int z, long long g, int n) {
            prolong_row<T>(F, C, eb, r, t, oh2, x, y, z, g, n);
        });
        return;
    }
    const long long sy = F.nx, sz = (long long)F.nx * F.ny;
    const T d = oh2 * T(1.0 / 6.0);
    const int ze = P.z0 & ~1, nzp = (P.z1 - ze + 1) >> 1;   // z pairs that meet the tile (it may start on an odd plane)
    for (int w = linear_tid(); w < 8 * (kTileY / 2) * nzp; w += 256) {
        const int xg = w & 7, rest = w >> 3;
        const int yp = rest % (kTileY / 2), zp = rest / (kTileY / 2);
        const int x = P.x0 + 4 * xg, y = P.y0 + 2 * yp, z = ze + 2 * zp;
        if (x >= F.nx || y >= F.ny) continue;
        if (y + 1 >= F.ny || z < P.z0 || z + 1 >= P.z1) {   // ragged edge: row by row
            for (int c = 0; c < 2; ++c)
                for (int b = 0; b < 2; ++b)
                    if (y + b < F.ny && z + c >= P.z0 && z + c < P.z1)
                        prolong_row<T>(F, C, eb, r, t, oh2, x, y + b, z + c,
                                       P.base + (z + c) * sz + (y + b) * sy + x, 4);
            continue;
        }
        const int I = x >> 1, J = y >> 1, K = z >> 1;
        // coarse rows (J-1+a, K-1+c), a, c in {0, 1}: values I-1, I, I+1
        T E[2][2][3];
#pragma unroll
        for (int c = 0; c < 2; ++c)
#pragma unroll
            for (int a = 0; a < 2; ++a) {
                const int JJ = J - 1 + a, KK = K - 1 + c;
                const bool ok = JJ >= 0 && JJ < C.ny && KK >= 0 && KK < C.nz;
                const T* row = eb + ((long long)(ok ? KK : 0) * C.ny + (ok ? JJ : 0)) * C.nx;
                E[c][a][0] = (ok && I >= 1) ? row[I - 1] : T(0);
                E[c][a][1] = ok ? row[I] : T(0);
                E[c][a][2] = ok ? row[I + 1] : T(0);
            }
        float4 rv[2][2];
#pragma unroll
        for (int c = 0; c < 2; ++c)
#pragma unroll
            for (int b = 0; b < 2; ++b)
                rv[c][b] = *reinterpret_cast<const float4*>(r + P.base + (z + c) * sz + (y + b) * sy + x);
        // x-interpolated coarse rows
        T X[2][2][4];
#pragma unroll
        for (int c = 0; c < 2; ++c)
#pragma unroll
            for (int a = 0; a < 2; ++a) {
                X[c][a][0] = T(0.5) * (E[c][a][0] + E[c][a][1]);
                X[c][a][1] = E[c][a][1];
                X[c][a][2] = T(0.5) * (E[c][a][1] + E[c][a][2]);
                X[c][a][3] = E[c][a][2];
            }
        // even fine index: 1/2 of coarse index - 1 and 1/2 of it; odd: the coarse index
#pragma unroll
        for (int c = 0; c < 2; ++c)
#pragma unroll
            for (int b = 0; b < 2; ++b) {
                T u[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const T y0 = b ? X[0][1][k] : T(0.5) * (X[0][0][k] + X[0][1][k]);   // plane K-1
                    const T y1 = b ? X[1][1][k] : T(0.5) * (X[1][0][k] + X[1][1][k]);   // plane K
                    u[k] = c ? y1 : T(0.5) * (y0 + y1);
                }
                const float4 v = rv[c][b];
                float4 o;
                o.x = d * v.x + u[0];
                o.y = d * v.y + u[1];
                o.z = d * v.z + u[2];
                o.w = d * v.w + u[3];
                *reinterpret_cast<float4*>(t + P.base + (z + c) * sz + (y + b) * sy + x) = o;
            }
    }
}

// e = t + omega D^-1 (r - A2 t) = (1 - omega) t + (omega/dd)(h^2 r + sum_nbr t);
// on level 0 also z.r per orbital -> rz, beta = rz / rz_old.
template <class T, bool kLevel0>
__global__ void __launch_bounds__(256) k_mg_postsmooth(const BlkDesc* __restrict__ blk, const LvlDesc* __restrict__ L,
                                                       const int4* __restrict__ tiles, const int* __restrict__ orb_blk,
                                                       const int* __restrict__ active, const T* __restrict__ r,
                                                       const T* __restrict__ t, T* __restrict__ e, T omega,
                                                       CgState st) {
    constexpr int V = Vec<T>::n;
    using VT = typename Vec<T>::type;
    __shared__ double scratch[32];
    const TilePos P = tile_pos(blk, L, tiles, orb_blk, blockIdx.x);
    const LvlDesc& D = L[P.b];
    if (!active[P.o] || D.fused) return;
    const T h2 = T(D.h * D.h);
    T rz = T(0);   // per-thread partial in the working precision; tile sums in float64
    tile_rows<T>(D, P, [&](int x, int y, int z, long long g, int n) {
        T c[V], nb[V], rv[V], out[V];
        centre_nbr<T, V>(t, D, x, y, z, g, n, c, nb);
        if (n == V) {
            const VT v = *reinterpret_cast<const VT*>(r + g);
#pragma unroll
            for (int k = 0; k < V; ++k) rv[k] = reinterpret_cast<const T*>(&v)[k];
        } else {
            rv[0] = r[g];
        }
        const bool edge = !kLevel0 && D.corr && (x + n >= D.nx || y == D.ny - 1 || z == D.nz - 1);
#pragma unroll
        for (int k = 0; k < V; ++k) {
            const T w = edge ? inv_diag<T>(D, x + k, y, z) : T(1.0 / 6.0);
            out[k] = (T(1) - omega) * c[k] + omega * w * (h2 * rv[k] + nb[k]);
            if (kLevel0 && k < n) rz += rv[k] * out[k];
        }
        store_n<T, V>(e + g, out, n);
    });
    if (kLevel0) {
        if (tile_arrive(rz, st.part, blockIdx.x, st.count + P.o, D.ntile, scratch)) {
            const double v = tile_gather(st.part, P.first, D.ntile, scratch);
            if (linear_tid() == 0) {
                st.count[P.o] = 0;
                const double old = st.rz[P.o];
                st.beta[P.o] = (old != 0.0) ? v / old : 0.0;
                st.rz[P.o] = v;
            }
        }
    }
}

// The coarse part of the V-cycle, from each block's first fused level down to
// its coarsest (40 damped-Jacobi sweeps from zero) and back up, one CTA per
// orbital with every level in shared memory: two arrays per level with a
// border of zeros (one point past each row, one row past each plane and a plane
// on either side, so that every neighbour of a point may be read); r, which
// becomes the level's correction e in place, and the smoothed residual, later
// the prolonged iterate.  When the first fused level
// is level 0 this is the whole preconditioner and the CTA also forms rz and beta.
//
// What bounds it: latency (a few thousand points, a barrier between the
// passes); in float64 one SM's 1.7 FMA per cycle.  A launch per pass spent
// 5 to 9 us on each level's four kernels whatever the level's size: at 64^3 x 10
// (levels of 16^3, 8^3 and 4^3 points) 54 us per V-cycle, here 20; at
// 40^3 x 5 in float64 (10^3 and 5^3) 55, here 37 us.
constexpr int kMgThreads = 1024;

template <class T>
struct MgSm {   // one level in shared memory
    int nx, ny, nz, px, pxy, G, corr;
    T h2;
    const T* w;       // [8] 1 / dd by the dimensions in which the point is last
    T *r, *s;         // first interior point of the bordered arrays
};

// inverse diagonal weight at (x, y, z)
template <class T>
__device__ __forceinline__ T mg_w(const MgSm<T>& M, int x, int y, int z) {
    return M.w[(x == M.nx - 1 ? 1 : 0) | (y == M.ny - 1 ? 2 : 0) | (z == M.nz - 1 ? 4 : 0)];
}
template <class T>
__device__ __forceinline__ T mg_nbr(const T* u, const MgSm<T>& M) {
    return ((u[-1] + u[1]) + (u[-M.px] + u[M.px])) + (u[-M.pxy] + u[M.pxy]);
}
template <class T, class Body>
__device__ __forceinline__ void mg_points(const MgSm<T>& M, Body body) {
    const int pl = M.nx * M.ny;
    for (int k = threadIdx.x; k < M.G; k += kMgThreads) {
        const int z = k / pl, rem = k - z * pl, y = rem / M.nx, x = rem - y * M.nx;
        body(k, x, y, z, z * M.pxy + y * M.px + x);
    }
}

template <class T>
__global__ void __launch_bounds__(kMgThreads) k_mg_coarse(const BlkDesc* __restrict__ blk, MgPtrs<T> mp,
                                                          const int* __restrict__ orb_blk, const int* __restrict__ active,
                                                          T omega, int nsweep, CgState st) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T* const sh = reinterpret_cast<T*>(smem_raw);
    __shared__ double scratch[32];
    __shared__ MgSm<T> lv[kMaxLevels];
    __shared__ T s_w[kMaxLevels][8];
    __shared__ int s_total;
    const int o = blockIdx.x, tid = threadIdx.x;
    if (!active[o]) return;
    const int b = orb_blk[o];
    const int f = mp.fused_level[b], lc = mp.coarsest_level[b];
    const int i = o - blk[b].orb0;
    if (tid == 0) {
        int at = 0;
        for (int l = f; l <= lc; ++l) {
            const LvlDesc& D = mp.lvl[l][b];
            MgSm<T>& M = lv[l];
            M.nx = D.nx; M.ny = D.ny; M.nz = D.nz;
            M.px = D.nx + 1;
            M.pxy = M.px * (D.ny + 1);
            M.G = (int)D.G;
            M.corr = D.corr;
            M.h2 = T(D.h * D.h);
            M.w = s_w[l];
            s_w[l][0] = T(1.0 / 6.0);
            for (int m = 1; m < 8; ++m) s_w[l][m] = T(D.idd[m]);
            const int pad = M.pxy * (D.nz + 2) + M.px + 1;
            M.r = sh + at + M.pxy + M.px + 1;
            M.s = M.r + pad;
            at += 2 * pad;
        }
        s_total = at;
    }
    __syncthreads();
    for (int k = tid; k < s_total; k += kMgThreads) sh[k] = T(0);
    __syncthreads();
    const LvlDesc& F = mp.lvl[f][b];
    const long long base = F.off + (long long)i * F.G;
    {
        const T* r = mp.r[f] + base;
        mg_points(lv[f], [&](int k, int, int, int, int q) { lv[f].r[q] = r[k]; });
    }
    __syncthreads();
    for (int l = f; l < lc; ++l) {
        const MgSm<T> M = lv[l];
        const MgSm<T> C = lv[l + 1];
        // s = r - A2 (omega D^-1 r)
        mg_points(M, [&](int, int x, int y, int z, int q) {
            const T* u = M.r + q;
            T sum;
            if (M.corr && (x >= M.nx - 2 || y >= M.ny - 2 || z >= M.nz - 2)) {   // a neighbour may lie on a last point
                sum = u[-1] * mg_w(M, x - 1, y, z) + u[1] * mg_w(M, x + 1, y, z) + u[-M.px] * mg_w(M, x, y - 1, z) +
                      u[M.px] * mg_w(M, x, y + 1, z) + u[-M.pxy] * mg_w(M, x, y, z - 1) +
                      u[M.pxy] * mg_w(M, x, y, z + 1);
            } else {
                sum = M.w[0] * mg_nbr(u, M);
            }
            M.s[q] = (T(1) - omega) * u[0] + omega * sum;
        });
        __syncthreads();
        // full weighting: coarse point I on fine point 2 I + 1
        mg_points(C, [&](int, int x, int y, int z, int q) {
            const T* u = M.s + (2 * z + 1) * M.pxy + (2 * y + 1) * M.px + 2 * x + 1;
            T acc = T(0);
#pragma unroll
            for (int c = -1; c <= 1; ++c)
#pragma unroll
                for (int a = -1; a <= 1; ++a) {
                    const T* v = u + c * M.pxy + a * M.px;
                    acc += (T(c == 0 ? 0.5 : 0.25) * T(a == 0 ? 0.5 : 0.25)) * (T(0.25) * (v[-1] + v[1]) + T(0.5) * v[0]);
                }
            C.r[q] = acc;
        });
        __syncthreads();
    }
    {   // coarsest level: the threads that own points (at most two each) meet at a barrier of their own warps
        const MgSm<T> M = lv[lc];
        static_assert(2 * kMgThreads >= kCoarseMax, "points per thread");
        const int nw = (min(M.G, kMgThreads) + 31) & ~31;
        if (tid < nw) {
            int q[2] = {0, 0};
            T c1[2] = {T(0), T(0)}, c2[2] = {T(0), T(0)};
            const int pl = M.nx * M.ny;
            const int np = tid + kMgThreads < M.G ? 2 : (tid < M.G ? 1 : 0);
#pragma unroll
            for (int a = 0; a < 2; ++a)
                if (a < np) {
                    const int k = tid + a * kMgThreads, z = k / pl, rem = k - z * pl, y = rem / M.nx, x = rem - y * M.nx;
                    q[a] = z * M.pxy + y * M.px + x;
                    c2[a] = omega * mg_w(M, x, y, z);
                    c1[a] = c2[a] * M.h2 * M.r[q[a]];
                }
            T *ea = M.s, *eb = M.r;   // (r is in the registers now; only its owner reads it)
#pragma unroll
            for (int a = 0; a < 2; ++a)
                if (a < np) ea[q[a]] = c1[a];
            for (int sw = 1; sw < nsweep; ++sw) {
                asm volatile("bar.sync 1, %0;" ::"r"(nw) : "memory");
#pragma unroll
                for (int a = 0; a < 2; ++a)
                    if (a < np) eb[q[a]] = c2[a] * mg_nbr(ea + q[a], M) + ((T(1) - omega) * ea[q[a]] + c1[a]);
                T* t = ea; ea = eb; eb = t;
            }
            if (ea != M.r) {
#pragma unroll
                for (int a = 0; a < 2; ++a)
                    if (a < np) M.r[q[a]] = ea[q[a]];
            }
        }
        __syncthreads();
    }
    const T* const r0 = mp.r[f] + base;
    T* const e0 = mp.e[f] + base;
    double rz = 0.0;
    for (int l = lc - 1; l >= f; --l) {
        const MgSm<T> M = lv[l];
        const MgSm<T> C = lv[l + 1];
        // t = omega D^-1 r + P e_c: per direction an odd point sits on coarse point
        // (x - 1) / 2, an even one halfway between x / 2 - 1 and x / 2
        mg_points(M, [&](int, int x, int y, int z, int q) {
            const int x1 = x >> 1, x0 = x1 - 1 + (x & 1);
            const int y1 = y >> 1, y0 = y1 - 1 + (y & 1);
            const int z1 = z >> 1, z0 = z1 - 1 + (z & 1);
            const T* p00 = C.r + z0 * C.pxy + y0 * C.px;
            const T* p01 = C.r + z0 * C.pxy + y1 * C.px;
            const T* p10 = C.r + z1 * C.pxy + y0 * C.px;
            const T* p11 = C.r + z1 * C.pxy + y1 * C.px;
            const T u = T(0.125) * (((p00[x0] + p00[x1]) + (p01[x0] + p01[x1])) + ((p10[x0] + p10[x1]) + (p11[x0] + p11[x1])));
            M.s[q] = omega * M.h2 * (M.corr ? mg_w(M, x, y, z) : M.w[0]) * M.r[q] + u;
        });
        __syncthreads();
        // e = t + omega D^-1 (r - A2 t), in place of r (read by its own point only)
        mg_points(M, [&](int k, int x, int y, int z, int q) {
            const T* t = M.s + q;
            const T w = M.corr ? mg_w(M, x, y, z) : M.w[0];
            const T e = (T(1) - omega) * t[0] + omega * w * (M.h2 * M.r[q] + mg_nbr(t, M));
            if (l > f) M.r[q] = e;
            else e0[k] = e;
            if (l == 0) rz += (double)M.r[q] * (double)e;
        });
        __syncthreads();
    }
    if (f == lc)   // a single fused level: the sweeps' result
        mg_points(lv[f], [&](int k, int, int, int, int q) {
            const T e = lv[f].r[q];
            if (f == 0) rz += (double)r0[k] * (double)e;
            e0[k] = e;
        });
    if (f == 0) {
        rz = block_sum(rz, scratch);
        if (tid == 0) {
            const double old = st.rz[o];
            st.beta[o] = (old != 0.0) ? rz / old : 0.0;
            st.rz[o] = rz;
        }
    }
}

// Elements of shared memory that k_mg_coarse needs for nlev levels from sides nx, ny, nz on
long long mg_coarse_elems(int nx, int ny, int nz, int nlev) {
    long long n = 0;
    for (int l = 0; l < nlev; ++l) {
        const long long px = (nx >> l) + 1, pxy = px * ((ny >> l) + 1);
        n += 2 * (pxy * ((nz >> l) + 2) + px + 1);
    }
    return n;
}
cudaError_t setup_mg_coarse(const flosic_ctx* c) {
    return c->opt.precision == FLOSIC_FP64 ? ensure_dyn_smem((const void*)k_mg_coarse<double>, c->mg.coarse_smem)
                                           : ensure_dyn_smem((const void*)k_mg_coarse<float>, c->mg.coarse_smem);
}

template <class T>
void launch_vcycle(const flosic_ctx* c, const MgPtrs<T>& mp, const int* active, cudaStream_t s) {
    const Multigrid& M = c->mg;
    const T omega = T(0.8);
    const dim3 tb(kTileX, kTileY / 2);
    for (int l = 0; l < M.fused_max; ++l) {   // some block's level l is above its fused ones
        if (M.ntiles[l] > 0) {
            k_mg_resid_smooth<T><<<(unsigned)M.ntiles[l], tb, 0, s>>>(c->d_blk, M.d_lvl[l], M.d_tiles[l],
                                                                     c->d_orb_blk, active, mp.r[l], mp.t[l],
                                                                     omega); note_launch(c);
        }
        if (M.ntiles[l + 1] > 0) {
            k_mg_restrict<T><<<(unsigned)M.ntiles[l + 1], tb, 0, s>>>(c->d_blk, M.d_lvl[l + 1], M.d_lvl[l],
                                                                     M.d_tiles[l + 1], c->d_orb_blk, active,
                                                                     mp.t[l], mp.r[l + 1]); note_launch(c);
        }
    }
    k_mg_coarse<T><<<c->norb, kMgThreads, M.coarse_smem, s>>>(c->d_blk, mp, c->d_orb_blk, active, omega, kCoarseSweeps,
                                                              c->ws.cg); note_launch(c);
    for (int l = M.fused_max - 1; l >= 0; --l) {
        if (M.ntiles[l] == 0) continue;
        k_mg_prolong<T><<<(unsigned)M.ntiles[l], tb, 0, s>>>(c->d_blk, M.d_lvl[l], M.d_lvl[l + 1],
                                                            M.d_tiles[l], c->d_orb_blk, active, mp.r[l],
                                                            mp.e[l + 1], mp.t[l], omega); note_launch(c);
        if (l == 0)
            k_mg_postsmooth<T, true><<<(unsigned)M.ntiles[0], tb, 0, s>>>(
                c->d_blk, M.d_lvl[0], M.d_tiles[0], c->d_orb_blk, active, mp.r[0], mp.t[0], mp.e[0], omega,
                c->ws.cg);
        else
            k_mg_postsmooth<T, false><<<(unsigned)M.ntiles[l], tb, 0, s>>>(
                c->d_blk, M.d_lvl[l], M.d_tiles[l], c->d_orb_blk, active, mp.r[l], mp.t[l], mp.e[l], omega,
                c->ws.cg);
        note_launch(c);
    }
}

template void launch_vcycle<float>(const flosic_ctx*, const MgPtrs<float>&, const int*, cudaStream_t);
template void launch_vcycle<double>(const flosic_ctx*, const MgPtrs<double>&, const int*, cudaStream_t);

}  // namespace flosic
