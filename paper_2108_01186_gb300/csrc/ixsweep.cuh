// The 12th-order stencil (Sec. II.A: high-order centred finite differences) in
// integer weights, and the staging of its planes, shared by the refinement update
// and the mixed-precision Hamiltonian apply.
#pragma once
#include <cmath>

#include "internal.cuh"

namespace flosic {

// ---------------------------------------------------------------------------
// Integer weights.  The 12th-order weights of the second derivative (w_m =
// 2 (-1)^(m+1) (6!)^2 / (m^2 (6-m)! (6+m)!), w_0 = -2 sum w_m) are rationals
// whose common denominator is 831600, so W_m = 831600 w_m are integers and
// h^2 Delta_h u = (1 / 831600) sum_m W_m (sum of the six neighbours at
// distance m).  An integer field is summed and weighted without rounding: six
// values of at most 2^28 stay below 2^31, the weighted sum below 2^53.
// ---------------------------------------------------------------------------
constexpr long long kW12Den = 831600;

__host__ __device__ constexpr long long w12_fact(int n) { return n <= 1 ? 1 : n * w12_fact(n - 1); }
__host__ __device__ constexpr long long w12_num(int m) {   // 2 (6!)^2 831600, signed
    return (m % 2 == 1 ? 2 : -2) * w12_fact(6) * w12_fact(6) * kW12Den;
}
__host__ __device__ constexpr long long w12_den(int m) { return (long long)m * m * w12_fact(6 - m) * w12_fact(6 + m); }
// W_m for m >= 1; W_0 of the three-dimensional centre is 3 (-2 sum_m W_m)
__host__ __device__ constexpr long long w12_int(int m) { return w12_num(m) / w12_den(m); }
__host__ __device__ constexpr long long w12_centre3() {
    return -6 * (w12_int(1) + w12_int(2) + w12_int(3) + w12_int(4) + w12_int(5) + w12_int(6));
}
static_assert(w12_num(1) % w12_den(1) == 0 && w12_num(2) % w12_den(2) == 0 && w12_num(3) % w12_den(3) == 0 &&
                  w12_num(4) % w12_den(4) == 0 && w12_num(5) % w12_den(5) == 0 && w12_num(6) % w12_den(6) == 0,
              "831600 is a common denominator of the 12th-order weights");
static_assert(w12_centre3() > -(1LL << 24) && w12_int(1) < (1LL << 24), "weights exact in float32");

// Host check of the integer weights against the float64 ones the other
// stencils use (|W_m / 831600 - w_m| at rounding level).
inline bool ix_weights_match() {
    double w[kHalf + 1];
    stencil_weights(w);
    for (int m = 1; m <= kHalf; ++m)
        if (std::fabs((double)w12_int(m) / (double)kW12Den - w[m]) > 1e-15 * std::fabs(w[m])) return false;
    return std::fabs((double)w12_centre3() / (double)kW12Den - 3.0 * w[0]) <= 1e-15 * std::fabs(3.0 * w[0]);
}

// I + Lo as a float-float pair (|I| < 2^53): I + 2^53 (non-negative) in pieces
// of 23, 23 and 8 bits, each exact as a float by the 2^23 bias (integer and
// float additions only: a 64-bit conversion would run on the float64 pipe),
// the bias removed from the top piece.
__device__ __forceinline__ ff ix_to_ff_b(long long I, float Lo) {
    const unsigned long long M = (unsigned long long)I + (1ull << 53);
    const float f0 = __uint_as_float(0x4B000000u | ((unsigned)M & 0x7fffffu)) - 8388608.f;
    const float f1 = (__uint_as_float(0x4B000000u | ((unsigned)(M >> 23) & 0x7fffffu)) - 8388608.f) * 8388608.f;
    const float f2 = (__uint_as_float(0x4B000000u | (unsigned)(M >> 46)) - 8388736.f) * 70368744177664.f;
    const ff v = ff_two_sum(f2, f1);
    return ff_two_sum(v.h, (v.l + f0) + Lo);
}

// z-windows in registers: the z-loop is unrolled kZU times, step u's window of
// 13 planes in slots u .. u + 12, and moved down by kZU slots after the last
// (twice: more spills at 128 registers; 13 times, which moves nothing, no longer
// fits the instruction cache).
constexpr int kZU = 2, kQ = 2 * kHalf + kZU;
template <class Pt>
__device__ __forceinline__ void ix_shift(Pt (&q)[kQ]) {
#pragma unroll
    for (int j = 0; j < 2 * kHalf; ++j) q[j] = q[j + kZU];
}

// ---------------------------------------------------------------------------
// Staging of a tile's planes with their 6-point x/y halo by asynchronous
// copies: a thread copies up to three pairs of neighbouring points (x even
// relative to the tile) per plane and splits the pairs that it copied itself, in
// place (a pair of split points takes 16 bytes, its raw points at most as many),
// so a copy needs no barrier, and any alignment, odd side or periodic wrap will
// do.  A plane that serves only as z-taps needs no halo.  A ring of ten planes:
// z .. z + 6, each split once (a z-window's head is read from the newest), two
// more on their way, and the one before z that slower threads may still read.
// ---------------------------------------------------------------------------
constexpr int kIxPts = kPX * kPY;                    // points of a staged plane
constexpr int kIxPairs = kIxPts / 2;
constexpr int kIxU = (kIxPairs + 255) / 256;         // pairs per thread
constexpr int kIxRing = 10;
template <int kRing = kIxRing>
__device__ __forceinline__ int ix_slot(int s, int d) { return s + d >= kRing ? s + d - kRing : s + d; }   // d planes on

template <int kBytes>
__device__ __forceinline__ void cp_async(void* dst, const void* src, int bytes) {   // the rest of kBytes is zeroed
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src),
                 "n"(kBytes), "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }

struct IxStage {
    int off[kIxU];    // in-plane offset of each pair's first point
    unsigned fl;      // per pair, 8 bits: 1 exists, 2 in the tile itself, 4 / 8 first / second point inside, 16 second wraps
    __device__ __forceinline__ void init(const LvlDesc& D, const TilePos& P, int pitch, int tid) {
        fl = 0;
#pragma unroll
        for (int j = 0; j < kIxU; ++j) {
            const int e = tid + j * 256;
            off[j] = 0;
            if (e >= kIxPairs) continue;
            const int yy = e / (kPX / 2), xx = 2 * (e - yy * (kPX / 2));
            int px = P.x0 - kHalf + xx, p1 = px + 1, py = P.y0 - kHalf + yy;
            if (D.per & 1) {
                px = wrap_coord(px, D.nx);
                p1 = wrap_coord(p1, D.nx);
            }
            if (D.per & 2) py = wrap_coord(py, D.ny);
            const bool iny = py >= 0 && py < D.ny;
            unsigned f = 1;
            if (xx >= kHalf && xx < kHalf + kTileX && yy >= kHalf && yy < kHalf + kTileY) f |= 2;
            if (iny && px >= 0 && px < D.nx) f |= 4;
            if (iny && p1 >= 0 && p1 < D.nx) f |= 8;
            if (p1 != px + 1) f |= 16;
            off[j] = (f & 12) ? py * pitch + px : 0;
            fl |= f << (8 * j);
        }
    }
    // is pair j read by a tap (full: the plane is one of the tile's)?
    __device__ __forceinline__ bool wants(int j, bool full) const { return (fl >> (8 * j)) & (full ? 1u : 2u); }
    // the same where both points are inside or neither is, and always aligned to their pair
    template <class T>
    __device__ __forceinline__ void copy_pair(int j, void* to, const T* plane, bool okz) const {
        cp_async<2 * sizeof(T)>(to, plane + off[j], okz && (fl & (4u << (8 * j))) ? 2 * (int)sizeof(T) : 0);
    }
    // pair j of the plane to `to`; vec: the points are always neighbours and both aligned to their pair
    template <class T>
    __device__ __forceinline__ void copy(int j, void* to, const T* plane, bool okz, bool vec, int nx) const {
        T* const dst = static_cast<T*>(to);
        const unsigned f = okz ? fl >> (8 * j) : 0u;
        const int b0 = (f & 4) ? (int)sizeof(T) : 0, b1 = (f & 8) ? (int)sizeof(T) : 0;
        if (vec) {
            cp_async<2 * sizeof(T)>(dst, plane + (b0 ? off[j] : 0), b0 + b1);
        } else {
            cp_async<sizeof(T)>(dst, plane + (b0 ? off[j] : 0), b0);
            cp_async<sizeof(T)>(dst + 1, plane + (b1 ? off[j] + ((f & 16) ? 1 - nx : 1) : 0), b1);
        }
    }
};

}  // namespace flosic
