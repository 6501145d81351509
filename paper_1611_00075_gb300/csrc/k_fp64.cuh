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

// Home positions minus the shift of each stencil coordinate (-1, 0, 1): one column
// per atom of the block (per group of P lanes).
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
// binomial series of the residual), from a float32 seed; x not negative.  An x
// whose high word lies below seed_hi takes the library's forms: x = 0 (two atoms
// at one place: infinity) and anything below float32's normal range, which
// f32_bits cannot hold, or (kNoSeed) every x, where r_c^2 itself is far outside
// float32's comfortable range.
__device__ __forceinline__ double rcp_f64(double x, int seed_hi) {
    if (__double2hiint(x) < seed_hi) return 1.0 / x;
    const double y = f64_bits(rcp_fast(f32_bits(x)));
    const double e = fma(-x, y, 1.0);
    return fma(y, fma(e, e, e), y);
}
__device__ __forceinline__ double rsqrt_f64(double x, int seed_hi) {
    if (__double2hiint(x) < seed_hi) return 1.0 / sqrt(x);
    const double y = f64_bits(rsqrt_fast(f32_bits(x)));
    const double e = fma(-(x * y), y, 1.0);
    return fma(y * e, fma(e, 0.375, 0.5), y);
}

// The nine home coordinates of atom i in column threadIdx.x / P, by its P lanes
// (every lane of the warp calls it).
template <int P>
__device__ __forceinline__ void load_home64(const ForceArgs &a, int i, int part, Home64 *h) {
    const int col = threadIdx.x / P;
#pragma unroll
    for (int k0 = 0; k0 < 9; k0 += P) {
        const int k = k0 + part;
        if (P == 1 || k < 9) {
            const int c = k % 3, d = k / 3;  // component, shift d - 1
            const double r = reinterpret_cast<const double *>(a.xr + i)[c];
            (c == 0 ? h->x : (c == 1 ? h->y : h->z))[d][col] =
                r - (double)(d - 1) * (c == 0 ? a.g.w[0] : (c == 1 ? a.g.w[1] : a.g.w[2]));
        }
    }
    __syncwarp();
}

// body(j, ex, ey, ez, r2) for every pair of sorted atom i inside r_c that lane
// `part` of its P lanes owns; e = x_j - x_i.  qi: the float32 position of i.  The
// next pair's float64 position is loaded before the current pair's body runs: a
// body is a chain of some 14 dependent float64 instructions, and with one to four
// warps per SM quarter nothing else hides the load.
template <int P, class Body>
__device__ __forceinline__ void f64_pairs(const ForceArgs &a, const ShiftTab *sh, const Home64 *h,
                                          int i, int part, const float4 &qi, const Body &body) {
    const int nq = (min(a.ncount[i], a.cap) + 3) >> 2;
    const uint4 *lq = reinterpret_cast<const uint4 *>(a.nlist + list_group(i, a.cap)) + (i & 31);
    const float lo = a.fc.scr_lo, hi = a.fc.scr_hi;
    const int t = threadIdx.x / P;
    unsigned left = 0;  // accepted entries of the current quad, band ones also in bits 4-7
    uint4 e4 = make_uint4(0u, 0u, 0u, 0u);
    int q = part;
    // the next accepted entry; false when there is none
    auto next = [&](uint32_t &ent, bool &band) -> bool {
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
        if (left == 0) return false;
        const int k = __ffs((int)left) - 1;
        band = (left >> (k + 4)) & 1u;
        left &= ~(17u << k);
        ent = k == 0 ? e4.x : (k == 1 ? e4.y : (k == 2 ? e4.z : e4.w));
        return true;
    };
    uint32_t ent = 0;
    bool band = false;
    bool have = next(ent, band);
    double4 rj = a.xr[have ? (ent & kIndexMask) : (uint32_t)i];
    while (have) {
        const uint32_t en = ent;
        const bool bn = band;
        const double4 r = rj;
        have = next(ent, band);
        if (have) rj = a.xr[ent & kIndexMask];
        const int s = (int)(en >> kIndexBits);
        const int sz = (s * 57) >> 9, sy = ((s - 9 * sz) * 11) >> 5, sx = s - 9 * sz - 3 * sy;
        const double ex = r.x - h->x[sx][t], ey = r.y - h->y[sy][t], ez = r.z - h->z[sz][t];
        const double r2 = ex * ex + ey * ey + ez * ez;
        if (!bn || r2 < a.fc.rc2) body((int)(en & kIndexMask), ex, ey, ez, r2);
    }
}

// sum over an atom's P lanes (all lanes of the warp call it)
template <int P>
__device__ __forceinline__ double lanes_sum(double x) {
#pragma unroll
    for (int o = P / 2; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    return x;
}

// Stores and the velocity-Verlet epilogue of one atom from its lanes' sums: by one
// lane per component where four or more share the atom (every lane of the warp
// calls it).
template <int MODE, bool SPECIES, int P>
__device__ __forceinline__ void f64_finish(const ForceArgs &a, int i, int part, bool on, double fx,
                                           double fy, double fz, float qw, int store_f) {
    if constexpr (P >= 4) {
        const int c = part & 3;
        const SplitState st = load_split_state<MODE>(a, i, c, on && part < 4);
        fx = lanes_sum<P>(fx);
        fy = lanes_sum<P>(fy);
        fz = lanes_sum<P>(fz);
        split_epilogue<MODE, SPECIES>(a, i, c, on && part < 4, c == 0 ? fx : (c == 1 ? fy : fz), qw,
                                      st, store_f);
    } else {
        if (!on) return;
        const size_t n = (size_t)a.n;
        if (MODE == FM_STORE || store_f) {
            a.f[i] = fx;
            a.f[n + i] = fy;
            a.f[2 * n + i] = fz;
        }
        if (MODE != FM_STORE) vv_epilogue<MODE, SPECIES>(a, i, fx, fy, fz, qw);
    }
}

// Lanes per atom.  One lane's chain of about 55 bodies takes 85 us however few
// atoms there are (a warp's float64 instruction holds the pipe for about as
// long as its result takes), so small systems are split; a split costs the sum
// of the lanes' largest shares.  Measured (LJ, force launch, us) with
// 1 / 4 / 8 / 16 lanes: 864 atoms 85 / 30 / 21 / 16, 2,048 atoms
// 90 / 31 / 21 / 20, 2,916 atoms 90 / 31 / 27 / 25, 4,000 atoms
// 90 / 31 / 27 / 31, 6,912 atoms 90 / 39 / 34 / 43, 10,976 atoms 92 / 49 / 51 / 63, 32,000 atoms
// 108 / 103 / 125 / 156, 87,808 atoms 222 / 257 / 309 / 402 (one lane per atom
// and the plain loop: 150 us up to 32,000 atoms, 437 us at 87,808; without the
// early load of the next position and the epilogue by components 33 at 4,000
// atoms with 4 lanes, 181 instead of 170 at 55,296).
inline int f64_split(int64_t n) {
    return n <= 3072 ? 16 : (n <= 8192 ? 8 : (n <= 32768 ? 4 : 1));
}

}  // namespace mdg
