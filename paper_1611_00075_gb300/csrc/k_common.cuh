// k_common.cuh -- pieces shared by the force kernels: the argument block,
// the fused velocity-Verlet epilogue (Sec. 3.3) and per-step bookkeeping.
#pragma once

#include "md_internal.cuh"

namespace mdg {

// float32 partial sums cover kChunkQ quads (64 list entries) before they are
// added to the float64 accumulators
constexpr int kChunkQ = 16;

// 1/x and 1/sqrt(x) in one special-function instruction, within 1 ulp and
// 2^-22.9 relative.  The .ftz forms: __fdividef and rsqrtf without -ftz also hold
// for denormal and huge arguments, which no squared distance the cutoff accepts
// needs, and take longer: the pair kernels return the same bits as with those
// forms on every system measured, and whole runs got shorter: alloy 12.00 -> 11.43 ms, Sutton-Chen 34.8 -> 33.4, batch 15.42 -> 15.07,
// porous 9.8 M 71.3 -> 69.7, EAM 15.30 -> 15.11 (the cases' own step counts).
__device__ __forceinline__ float rcp_fast(float x) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ float rsqrt_fast(float x) {
    float r;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// Sum over the P neighbouring lanes that share an item (P a power of two; every
// lane of the warp calls it).
template <int P, class T>
__device__ __forceinline__ T split_sum(T x) {
#pragma unroll
    for (int o = P / 2; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    return x;
}

// A normal float32 as float64 by integer operations (the conversion instruction runs
// on the float64 pipe).
__device__ __forceinline__ bool normal_f32(float f) {
    return (__float_as_uint(f) & 0x7fffffffu) - 0x00800000u < 0x7f000000u;
}
__device__ __forceinline__ double widen_f32(float f) {
    const unsigned b = __float_as_uint(f);
    return __hiloint2double(
        (int)((((b & 0x7fffffffu) >> 3) + 0x38000000u) | (b & 0x80000000u)), (int)(b << 29));
}

// s + e = a + b exactly (Knuth's two-sum), s the rounded sum.
__device__ __forceinline__ void two_sum(float a, float b, float &s, float &e) {
    s = __fadd_rn(a, b);
    const float t = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, t)), __fsub_rn(b, t));
}

// The sums over an item's P lanes (4 or 8, aligned) of the float32 values x, y, z
// and e: the lane with part & 3 = 0, 1, 2, 3 returns that of x, y, z, e (every lane
// of the warp calls it).  The lanes' values are added as pairs of floats, 48 bits,
// and once in float64: what is rounded off is below 2^-45 of the largest partial
// sum, while each value carries float32's own rounding.  Each exchange halves what
// a lane still holds.  (Float64 additions wait for a pipe of 1/64 of the float32
// rate: one step of 16,384 atoms 17.5 us with them, 15.9 with plain float32 sums,
// 16.2 in this form; 864 atoms 9.6, 9.4 and 9.4.)
template <int P>
__device__ __forceinline__ double split_component(float x, float y, float z, float e, int part) {
    static_assert(P == 4 || P == 8, "one lane per component");
    constexpr unsigned full = 0xffffffffu;
    const bool hi = part & 2, lo = part & 1;
    float s0, r0, s1, r1, s, r;
    two_sum(hi ? z : x, __shfl_xor_sync(full, hi ? x : z, 2), s0, r0);
    two_sum(hi ? e : y, __shfl_xor_sync(full, hi ? y : e, 2), s1, r1);
    const float ss = __shfl_xor_sync(full, lo ? s0 : s1, 1);
    const float rr = __shfl_xor_sync(full, lo ? r0 : r1, 1);
    two_sum(lo ? s1 : s0, ss, s, r);
    r += (lo ? r1 : r0) + rr;
    if (P == 8) {
        const float s8 = __shfl_xor_sync(full, s, 4), r8 = __shfl_xor_sync(full, r, 4);
        float t;
        two_sum(s, s8, s, t);
        r += r8 + t;
    }
    // zero, infinity and NaN have no rest (nor has a denormal sum)
    if (!normal_f32(s)) return (double)s;
    return widen_f32(s) + (normal_f32(r) ? widen_f32(r) : 0.0);
}

// pair(entry) for every entry of the quads part, part + P, ... of an item's list
// (lq: its first quad; quads lie 32 apart), one quad loaded ahead.
template <int P, class Pair>
__device__ __forceinline__ void split_quads(const uint4 *lq, int nq, int part, const Pair &pair) {
    uint4 nxt = part < nq ? __ldcs(lq + (size_t)part * 32) : make_uint4(0u, 0u, 0u, 0u);
    for (int q = part; q < nq; q += P) {
        const uint4 e4 = nxt;
        if (q + P < nq) nxt = __ldcs(lq + (size_t)(q + P) * 32);
        pair(e4.x);
        pair(e4.y);
        pair(e4.z);
        pair(e4.w);
    }
}

struct ForceArgs {
    int n, cap, step, rebuild_every;
    const float4 *__restrict__ xq;
    float4 *__restrict__ xq_out;
    const double4 *__restrict__ xr;
    double4 *__restrict__ xr_out;
    const float4 *__restrict__ xq_build;
    double *__restrict__ v;
    double *__restrict__ f;
    double *__restrict__ e_atom;
    const uint32_t *__restrict__ nlist;
    const int32_t *__restrict__ ncount;
    double *__restrict__ rho;     // many-body: rho_i (Eq. 2)
    float *__restrict__ dF32;     // many-body: F'(rho_i) in float32
    float4 *__restrict__ xqf;     // many-body, mixed: (x, y, z, F'(rho)) per atom
    double *__restrict__ dF64;    // many-body: F'(rho_i) in float64
    const uint16_t *__restrict__ rep;     // batches: replica of each sorted atom
    const float4 *__restrict__ widths32;  // batches: float32 cell widths of each box
    DevStatus *ds;
    Grid g;
    ForceConsts fc;
};

// The stencil coordinates (-1, 0 or 1 per axis) of a list entry, whose top five
// bits hold 9 (z + 1) + 3 (y + 1) + (x + 1).  One funnel shift makes the float
// 2^23 + that number, and six additions and multiply-adds split it (every
// quotient is rounded to an integer by adding and subtracting 1.5 x 2^23; all of
// it is exact).  A pair kernel that reads the cell shift from a table in shared
// memory spends three of its 16 L1 wavefronts per entry on it, and L1 wavefronts
// are what these kernels are short of; the multiply-add that applies the shift
// (exactly: +-w or 0) replaces the addition of the table's value.
// Against the table, whole runs: 331 k atoms (per-atom lists) 5.28 -> 4.84 ms,
// liquid of 1 M 6.59 -> 6.13, 64 boxes 13.28 -> 12.32, Sutton-Chen 32.8 -> 31.1,
// EAM 14.28 -> 13.55, alloy 10.43 -> 10.06, porous 9.8 M 66.2 -> 64.0; same bits.
// (The same split in shifts and masks was slower than the table: they run on the
// half-rate pipe of the comparisons.)
__device__ __forceinline__ float3 stencil_of(uint32_t ent) {
    const float kRound = 12582912.f;
    const float c = __uint_as_float(__funnelshift_l(ent, 0x02580000u, 5)) - 8388621.f;
    const float z = fmaf(c, 1.f / 9.f, kRound) - kRound;
    const float r = fmaf(z, -9.f, c);
    const float y = fmaf(r, 1.f / 3.f, kRound) - kRound;
    return make_float3(fmaf(y, -3.f, r), y, z);
}
static_assert(kIndexBits == 27, "stencil_of's shift");

// |e|^2 in the rounding that every pass over the same pairs uses (left to the
// contraction rules, ex ex + ey ey + ez ez gave other bits in other kernels): one
// pair must not be inside r_c for one pass and outside for another.
__device__ __forceinline__ float dist2(float ex, float ey, float ez) {
    return fmaf(ez, ez, fmaf(ex, ex, ey * ey));
}

// The cell widths of replica r of a batch.
__device__ __forceinline__ float3 replica_width(const ForceArgs &a, int r) {
    const float4 w = a.widths32[r];
    return make_float3(w.x, w.y, w.z);
}

// Float32 cell shifts (dx, dy, dz) * w of the 27 stencil cells, in shared
// memory, one array per component: the lanes of a warp read up to 27
// distinct words of one array, which sit in 27 distinct banks, so each read
// is a single wavefront (a float4 table costs several).
struct ShiftTab {
    float x[32], y[32], z[32];
};

__device__ __forceinline__ void load_shifts_f32(const Grid &g, ShiftTab *sh) {
    if (threadIdx.x < kStencil) {
        int s = threadIdx.x;
        int dx = s % 3 - 1, dy = (s / 3) % 3 - 1, dz = s / 9 - 1;
        sh->x[s] = (float)(dx * g.w[0]);
        sh->y[s] = (float)(dy * g.w[1]);
        sh->z[s] = (float)(dz * g.w[2]);
    }
}

// Fills a ForceArgs from the handle for the current double-buffer index.
ForceArgs make_force_args(md_system *h);

// Shared epilogue: kick (and drift) of atom i with its float64 force.
// SPECIES: a multi-element system, whose atom takes its species' mass (a
// compile-time switch: a run-time test here cost the persistent kernel 6 %).
template <int MODE, bool SPECIES = false>
__device__ __forceinline__ void vv_epilogue(const ForceArgs &a, int i, double Fx, double Fy,
                                            double Fz, float qw) {
    const size_t n = (size_t)a.n;
    double im = a.fc.inv_m;
    if (SPECIES) im = pick4(a.fc.t_inv_m, species_of(__float_as_uint(qw)));
    const double hk = (MODE == FM_FUSED_FULL) ? a.fc.dt * im : 0.5 * a.fc.dt * im;
    double vx = a.v[i] + hk * Fx;
    double vy = a.v[n + i] + hk * Fy;
    double vz = a.v[2 * n + i] + hk * Fz;
    a.v[i] = vx;
    a.v[n + i] = vy;
    a.v[2 * n + i] = vz;
    if (MODE == FM_FUSED_FULL) {
        double4 r = a.xr[i];
        r.x += a.fc.dt * vx;
        r.y += a.fc.dt * vy;
        r.z += a.fc.dt * vz;
        a.xr_out[i] = r;
        float4 q = make_float4((float)r.x, (float)r.y, (float)r.z, qw);
        a.xq_out[i] = q;
        float4 b = a.xq_build[i];
        float ddx = q.x - b.x, ddy = q.y - b.y, ddz = q.z - b.z;
        float d2 = ddx * ddx + ddy * ddy + ddz * ddz;
        if (!(d2 <= 3.0e38f)) atomicCAS(&a.ds->status, 0, (int)MD_ERR_NONFINITE);
        if (a.rebuild_every <= 0 && d2 > a.fc.half_skin2f) a.ds->rebuild = 1;
    }
}

// What the epilogue of one component of an atom reads, loaded before its list is
// walked.
struct SplitState {
    double v, r;  // velocity and position component
    float b;      // position component at the last build
};
template <int MODE>
__device__ __forceinline__ SplitState load_split_state(const ForceArgs &a, int i, int c, bool on) {
    SplitState t{0.0, 0.0, 0.f};
    if (MODE != FM_STORE && on && c < 3) {
        t.v = a.v[(size_t)c * a.n + i];
        if (MODE == FM_FUSED_FULL) {
            t.r = reinterpret_cast<const double *>(a.xr + i)[c];
            t.b = reinterpret_cast<const float *>(a.xq_build + i)[c];
        }
    }
    return t;
}

// Stores and the velocity-Verlet epilogue of atom i by four neighbouring lanes
// (aligned to four; every lane of the warp calls it): lane c of the four owns
// component c (x, y, z), lane 3 the position word qw.  on: the atom exists.  The
// arithmetic of each component is vv_epilogue's; a float64 instruction then
// serves three components of eight atoms where one lane per atom would spend
// three on eight.
template <int MODE, bool SPECIES = false>
__device__ __forceinline__ void split_epilogue(const ForceArgs &a, int i, int c, bool on, double F,
                                               float qw, const SplitState &t, int store_f) {
    const size_t n = (size_t)a.n;
    const bool comp = on && c < 3;
    if ((MODE == FM_STORE || store_f) && comp) a.f[(size_t)c * n + i] = F;
    if (MODE == FM_STORE) return;
    double im = a.fc.inv_m;
    if (SPECIES) im = pick4(a.fc.t_inv_m, species_of(__float_as_uint(qw)));
    const double hk = (MODE == FM_FUSED_FULL) ? a.fc.dt * im : 0.5 * a.fc.dt * im;
    const double v = t.v + hk * F;
    if (comp) a.v[(size_t)c * n + i] = v;
    if (MODE != FM_FUSED_FULL) return;
    const double r = t.r + a.fc.dt * v;
    const float q = c < 3 ? (float)r : qw;
    if (comp) reinterpret_cast<double *>(a.xr_out + i)[c] = r;
    if (on) reinterpret_cast<float *>(a.xq_out + i)[c] = q;
    // the displacement since the last build, summed as in vv_epilogue
    const float dd = q - t.b;
    const int lane = (int)(threadIdx.x & 31) & ~3;
    const float dx = __shfl_sync(0xffffffffu, dd, lane), dy = __shfl_sync(0xffffffffu, dd, lane + 1),
                dz = __shfl_sync(0xffffffffu, dd, lane + 2);
    const float d2 = dx * dx + dy * dy + dz * dz;
    if (on && c == 0) {
        if (!(d2 <= 3.0e38f)) atomicCAS(&a.ds->status, 0, (int)MD_ERR_NONFINITE);
        if (a.rebuild_every <= 0 && d2 > a.fc.half_skin2f) a.ds->rebuild = 1;
    }
}

// Lanes per work item (atom or two-atom slot) of the mixed passes: one item's
// list is a serial chain of gathers, so a system that leaves most of the GPU
// idle is split.  The lanes' float32 sums cover at most cap / P entries, kept
// within the 64 of the one-lane kernels' chunks; per-atom rows add them as
// pairs of floats (split_component), where one lane adds its chunks in float64;
// slots add in float32, as one lane does.
// One step (LJ, replayed, disordered fcc), us.  Four lanes end where one lane takes
// the same time: per-atom rows, four / one, 17.6 / 19.6 at 42,592 atoms, 19.7 / 20.1
// at 46,552, 20.1 / 19.7 at 48,668, 21.2 / 20.2 at 55,296; slots of two, by atoms,
// 26.6 / 30.5 at 87,808, 32.6 / 32.6 at 119,164, 34.6 / 34.4 at 131,072.  Eight lanes
// against four: rows 9.9 / 11.4 at 864 atoms, 11.7 / 11.9 at 5,324, 13.0 / 12.5 at
// 8,788, 16.0 / 14.8 at 16,384; slots 11.7 / 13.0 at 864, 13.7 / 14.0 at 13,500,
// 19.9 / 17.6 at 32,000.  They go past the crossing (6,000 atoms, 7,000 slots) because
// lanes set the order of an item's sums: a batch moves its boxes bit for bit as they
// move alone only while the batch and each box have the same lanes.
constexpr int64_t kEightLanes = 16384, kFourLanesAtoms = 47104, kFourLanesSlots = 61440;
inline int mixed_split(int64_t items, int cap, int64_t four) {
    if (items <= kEightLanes && cap <= 8 * 4 * kChunkQ) return 8;
    if (items <= four && cap <= 4 * 4 * kChunkQ) return 4;
    return 1;
}
// Eight lanes or one, for the passes with more work per entry; each says its limit.
// Two-species LJ, one step with eight lanes against one, us: per-atom lists 12.7 /
// 21.5 at 2,048 atoms, 22.1 / 24.1 at 32,000; slots of two 14.5 / 29 at 10,976
// atoms, 30.8 / 33.5 at 70,304, 47.6 / 38.5 at 131,072.
constexpr int64_t kTypedSplit = 32768;
inline int split8(int64_t items, int cap, int64_t limit) {
    return items <= limit && cap <= 8 * 4 * kChunkQ ? 8 : 1;
}

// Adds v over the converged lanes of the warp to the in-cutoff pair counter
// (correct for any subset of lanes: each group's leader adds its own sum).
__device__ __forceinline__ void count_pairs(DevStatus *ds, unsigned v) {
    const unsigned m = __activemask();
    const unsigned t = __reduce_add_sync(m, v);
    if ((int)(threadIdx.x & 31) == __ffs(m) - 1) atomicAdd(&ds->pairs_cut, (unsigned long long)t);
}

template <int MODE>
__device__ __forceinline__ void step_bookkeeping(const ForceArgs &a) {
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        if (MODE == FM_FUSED_FULL) {
            a.ds->abs_fresh = 0;
            int sb = a.ds->since_build + 1;
            a.ds->since_build = sb;
            if (a.rebuild_every > 0 && sb >= a.rebuild_every) a.ds->rebuild = 1;
        }
        // a device-side count, so that a step replayed from a CUDA graph counts too
        if (MODE != FM_STORE) a.ds->steps_done += 1;
    }
}

}  // namespace mdg
