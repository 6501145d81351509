// k_fp64.cuh -- the pair loop of the float64 passes.
//
// GB300's float64 pipe runs at 1/64 of the float32 rate, so a float64 pass costs
// what its float64 instructions cost and the rest is nearly free.  The loop
// therefore
//   - decides in float32 which list entries can lie inside r_c (a band around
//     r_c^2 is decided in float64), and runs the float64 body for those only:
//     a lane walks its quads by itself until it has an accepted entry, so a
//     warp's body count is its largest number of pairs inside r_c, not its
//     longest list;
//   - takes the home position already moved against the stencil cell's shift
//     (nine numbers per atom in shared memory): three subtractions per pair;
//   - starts 1/x and 1/sqrt(x) from the float32 special function and refines
//     (one step of third order: the seed's relative error of 2^-22 becomes
//     2^-64, below float64's rounding), three and five instructions instead of
//     the dozen or more of a division or a square root.
// About 17 float64 instructions per pair inside r_c for Lennard-Jones, where
// the plain loop ran 30 to 47 per list entry.
//
// P lanes (a power of two, neighbours in a warp) share an atom and take every
// P-th quad of its list; f64_split says how many.
#pragma once

#include "k_common.cuh"

namespace mdg {

constexpr int kF64Block = 128;

// Home positions minus the shift of each stencil coordinate (-1, 0, 1).
struct Home64 {
    double x[3][kF64Block], y[3][kF64Block], z[3][kF64Block];
};

// float32 of a positive normal double in float32's range, rounded toward zero,
// and back, both by integer operations (the conversion instructions run on the
// float64 pipe)
__device__ __forceinline__ float f32_bits(double d) {
    const unsigned hi = (unsigned)__double2hiint(d), lo = (unsigned)__double2loint(d);
    return __uint_as_float(((hi - 0x38000000u) << 3) | (lo >> 29));
}
__device__ __forceinline__ double f64_bits(float f) {
    const unsigned b = __float_as_uint(f);
    return __hiloint2double((int)((b >> 3) + 0x38000000u), (int)(b << 29));
}

// 1/x (Newton's iteration with its second-order term) and 1/sqrt(x) (the
// binomial series of the residual), from a float32 seed; x positive.  seeded =
// false (r_c^2 far outside float32's comfortable range): the library's forms.
__device__ __forceinline__ double rcp_f64(double x, bool seeded) {
    if (!seeded) return 1.0 / x;
    const double y = f64_bits(rcp_fast(f32_bits(x)));
    const double e = fma(-x, y, 1.0);
    return fma(y, fma(e, e, e), y);
}
__device__ __forceinline__ double rsqrt_f64(double x, bool seeded) {
    if (!seeded) return 1.0 / sqrt(x);
    const double y = f64_bits(rsqrt_fast(f32_bits(x)));
    const double e = fma(-(x * y), y, 1.0);
    return fma(y * e, fma(e, 0.375, 0.5), y);
}

// The nine home coordinates of atom i, in the calling thread's column.
__device__ __forceinline__ void load_home64(const ForceArgs &a, int i, Home64 *h) {
    const double4 r = a.xr[i];
#pragma unroll
    for (int d = -1; d <= 1; ++d) {
        h->x[d + 1][threadIdx.x] = r.x - d * a.g.w[0];
        h->y[d + 1][threadIdx.x] = r.y - d * a.g.w[1];
        h->z[d + 1][threadIdx.x] = r.z - d * a.g.w[2];
    }
}

// body(j, ex, ey, ez, r2) for every pair of sorted atom i inside r_c that lane
// `part` of its P lanes owns; e = x_j - x_i.  qi: the float32 position of i.
template <int P, class Body>
__device__ __forceinline__ void f64_pairs(const ForceArgs &a, const ShiftTab *sh, const Home64 *h,
                                          int i, int part, const float4 &qi, const Body &body) {
    const int nq = (min(a.ncount[i], a.cap) + 3) >> 2;
    const uint4 *lq = reinterpret_cast<const uint4 *>(a.nlist + list_group(i, a.cap)) + (i & 31);
    const float lo = a.fc.scr_lo, hi = a.fc.scr_hi;
    const int t = threadIdx.x;
    unsigned left = 0;  // accepted entries of the current quad, band ones also in bits 4-7
    uint4 e4 = make_uint4(0u, 0u, 0u, 0u);
    int q = part;
    for (;;) {
        while (left == 0 && q < nq) {
            e4 = __ldcs(lq + (size_t)q * 32);
            q += P;
            const uint32_t ents[4] = {e4.x, e4.y, e4.z, e4.w};
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const float4 qj = __ldg(a.xq + (ents[k] & kIndexMask));
                const uint32_t st = ents[k] >> kIndexBits;
                const float ex = (qj.x - qi.x) + sh->x[st], ey = (qj.y - qi.y) + sh->y[st],
                            ez = (qj.z - qi.z) + sh->z[st];
                const float r2 = ex * ex + ey * ey + ez * ez;
                // written so that a NaN (lo and hi are NaN when float32 cannot
                // decide) goes to the float64 test
                if (!(r2 >= hi)) left |= (r2 < lo ? 1u : 17u) << k;
            }
        }
        if (left == 0) break;
        const int k = __ffs((int)left) - 1;
        const bool band = (left >> (k + 4)) & 1u;
        left &= ~(17u << k);
        const uint32_t ent = k == 0 ? e4.x : (k == 1 ? e4.y : (k == 2 ? e4.z : e4.w));
        const int j = (int)(ent & kIndexMask);
        const int s = (int)(ent >> kIndexBits);
        const int sz = (s * 57) >> 9, sy = ((s - 9 * sz) * 11) >> 5, sx = s - 9 * sz - 3 * sy;
        const double4 rj = a.xr[j];
        const double ex = rj.x - h->x[sx][t], ey = rj.y - h->y[sy][t], ez = rj.z - h->z[sz][t];
        const double r2 = ex * ex + ey * ey + ez * ez;
        if (band && !(r2 < a.fc.rc2)) continue;
        body(j, ex, ey, ez, r2);
    }
}

// sum over an atom's P lanes (all lanes of the warp call it)
template <int P>
__device__ __forceinline__ double lanes_sum(double x) {
#pragma unroll
    for (int o = P / 2; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    return x;
}

// Lanes per atom.  One lane's chain of about 55 bodies takes 85 us however few
// atoms there are (a warp's float64 instruction holds the pipe for about as
// long as its result takes), so small systems are split; a split costs the sum
// of the lanes' largest shares.  Measured (LJ, force launch, us) with 1 / 4 / 16
// lanes: 864 atoms 86 / 32 / 18, 4,000 atoms 90 / 33 / 32, 6,912 atoms
// 90 / 40 / 45, 19,652 atoms 101 / 76 / 107, 32,000 atoms 108 / 104 / 167,
// 87,808 atoms 221 / 263 / 434 (one lane per atom and the plain loop: 150 us up
// to 32,000 atoms, 437 us at 87,808).
inline int f64_split(int64_t n) { return n <= 4096 ? 16 : (n <= 32768 ? 4 : 1); }

}  // namespace mdg
