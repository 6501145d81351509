// k_lj.cu -- Lennard-Jones forces from a full neighbour list (Sec. 2.2).
//
// Pair force F = -(1/d) dPhi/dr R with R = r_i - r_j; for the truncated and
// energy-shifted Lennard-Jones pair potential
//     Phi(r) = 4 eps [(s/r)^12 - (s/r)^6] - Phi(r_c),   r < r_c,
// -(1/d) dPhi/dr = 48 eps / d^2 [(s/d)^12 - (s/d)^6 / 2].
//
// With a full list every atom sums its own force (f_j is never written by
// the thread of atom i), which is how this kernel avoids the Newton's-third-
// law race of Sec. 1 without atomics.  One thread per sorted atom walks its
// list; the lanes of a warp read their k-th entries from one 128-byte line.
//
// Precision:
//   MIXED  the pair vector, r^2, 1/r^2, (s/r)^6 and the force scalar are
//          float32, computed from cell-relative float32 coordinates plus the
//          float32 cell shift of the entry's stencil cell (stencil_of); each chunk of
//          64 entries is summed in float32 and the chunk sums are added in
//          float64 (the GPU form of the paper's blocked pair loop; where lanes
//          share an atom, their sums of at most 64 entries as pairs of floats).  Entries
//          arrive four at a time (one 16-byte load), so four gathers are in
//          flight before the arithmetic that needs them.
//   FP64   everything in float64 (the plain path).
//
// Modes (ForceMode): FM_STORE writes forces; FM_FUSED_FULL also applies the
// two merged half kicks of consecutive velocity-Verlet steps (v += dt f / m)
// and the drift (x += dt v) of the atom, writing its position into the other
// buffer of a double-buffered pair; FM_FUSED_HALF applies the closing half
// kick (v += dt f / 2m).  The drift also measures the displacement since the
// last list build and raises the rebuild flag past half the skin (Sec. 3.3).
#include <type_traits>

#include "k_fp64.cuh"
#include "k_pair.cuh"

namespace mdg {

// The whole per-atom job of the mixed path for sorted atom i: pair loop over
// its list, stores, and the velocity-Verlet epilogue.  MULTI (systems of
// several boxes) takes the cell widths of the atom's own box.  P > 1: the P
// lanes of the atom (this one is `part`; on: the atom exists) each walk every P-th
// quad and add their sums.  TABLE: the cell shifts come from sh (the same bits as
// computed ones).
template <int MODE, bool ENERGY, bool MULTI = false, int P = 1, bool TABLE = false>
__device__ __forceinline__ void lj_mixed_atom(const ForceArgs &a, int i, int store_f,
                                              int part = 0, bool on = true,
                                              const ShiftTab *sh = nullptr) {
    const float3 w = MULTI ? replica_width(a, (int)a.rep[i])
                           : make_float3(a.g.wf[0], a.g.wf[1], a.g.wf[2]);
    const float4 qi = a.xq[i];
    const int nq = (min(a.ncount[i], a.cap) + 3) >> 2;
    const uint4 *lq = reinterpret_cast<const uint4 *>(a.nlist + list_group(i, a.cap)) + (i & 31);
    const float rc2 = a.fc.rc2f, sig2 = a.fc.sig2f, e48 = a.fc.eps48f;
    double Fx = 0.0, Fy = 0.0, Fz = 0.0, E = 0.0;
    unsigned npair = 0;
    float fx = 0.f, fy = 0.f, fz = 0.f, e = 0.f;
    auto pair = [&](uint32_t ent) {
        const float4 qj = __ldg(a.xq + (ent & kIndexMask));
        float ex, ey, ez;
        if (TABLE) {
            const uint32_t st = ent >> kIndexBits;
            ex = (qj.x - qi.x) + sh->x[st];
            ey = (qj.y - qi.y) + sh->y[st];
            ez = (qj.z - qi.z) + sh->z[st];
        } else {
            const float3 st = stencil_of(ent);
            ex = fmaf(st.x, w.x, qj.x - qi.x);
            ey = fmaf(st.y, w.y, qj.y - qi.y);
            ez = fmaf(st.z, w.z, qj.z - qi.z);
        }
        const float r2 = dist2(ex, ey, ez);
        if (r2 < rc2) {
            const float r2i = rcp_fast(r2);
            float s6 = sig2 * r2i;
            s6 = s6 * s6 * s6;
            const float fs = e48 * r2i * s6 * (s6 - 0.5f);
            fx -= fs * ex;
            fy -= fs * ey;
            fz -= fs * ez;
            if (ENERGY) {
                e += a.fc.eps4f * s6 * (s6 - 1.0f) - a.fc.shiftf;
                ++npair;
            }
        }
    };
    if constexpr (P > 1) {
        // the float32 sums cover a P-th of the list, at most a chunk's 64 entries
        const int c = part & 3;
        const SplitState t = load_split_state<MODE>(a, i, c, on && part < 4);
        split_quads<P>(lq, on ? nq : 0, part, pair);
        const double F = split_component<P>(fx, fy, fz, e, part);
        if (ENERGY) {
            if (on) count_pairs(a.ds, npair);
            if (on && part == 3) a.e_atom[i] = 0.5 * F;
        }
        split_epilogue<MODE>(a, i, c, on && part < 4, F, qi.w, t, store_f);
        return;
    } else {
        // list quads stream through once (evict-first), one quad loaded ahead;
        // the float64 sums run once per chunk, outside the inner loop
        uint4 nxt = nq > 0 ? __ldcs(lq) : make_uint4(0u, 0u, 0u, 0u);
        for (int q0 = 0; q0 < nq; q0 += kChunkQ) {
            const int q1 = min(q0 + kChunkQ, nq);
            for (int q = q0; q < q1; ++q) {
                const uint4 e4 = nxt;
                if (q + 1 < nq) nxt = __ldcs(lq + (size_t)(q + 1) * 32);
                pair(e4.x);
                pair(e4.y);
                pair(e4.z);
                pair(e4.w);
            }
            Fx += (double)fx;
            Fy += (double)fy;
            Fz += (double)fz;
            fx = fy = fz = 0.f;
            if (ENERGY) {
                E += (double)e;
                e = 0.f;
            }
        }
    }
    const size_t n = (size_t)a.n;
    if (MODE == FM_STORE || store_f) {
        a.f[i] = Fx;
        a.f[n + i] = Fy;
        a.f[2 * n + i] = Fz;
    }
    if (ENERGY) {
        a.e_atom[i] = 0.5 * E;
        count_pairs(a.ds, npair);
    }
    if (MODE != FM_STORE) vv_epilogue<MODE>(a, i, Fx, Fy, Fz, qi.w);
}

// The whole per-atom job of the plain float64 path for sorted atom i, shared by
// P lanes (lane `part`); on: the atom exists (all lanes of a warp call this).
// The force scalar 48 eps r^-2 s6 (s6 - 1/2) with u = (sigma/r)^2 is
// (48 eps / r^2) u^3 (u^3 - 1/2).
template <int MODE, bool ENERGY, int P>
__device__ __forceinline__ void lj_fp64_atom(const ForceArgs &a, const ShiftTab *sh, Home64 *h,
                                             int i, int part, bool on, int store_f) {
    double fx = 0.0, fy = 0.0, fz = 0.0, e = 0.0;
    unsigned npair = 0;
    float qw = 0.f;
    load_home64<P>(a, i, part, h);
    if (on) {
        const float4 qi = a.xq[i];
        qw = qi.w;
        const double sig2 = a.fc.sig2, e48 = a.fc.eps48;
        const int seed_hi = a.fc.f64_seed_hi;
        f64_pairs<P>(a, sh, h, i, part, qi, [&](int, double ex, double ey, double ez, double r2) {
            const double r2i = rcp_f64(r2, seed_hi);
            double s6 = sig2 * r2i;
            s6 = s6 * s6 * s6;
            const double fs = (e48 * r2i) * fma(s6, s6, -0.5 * s6);
            fx -= fs * ex;
            fy -= fs * ey;
            fz -= fs * ez;
            if (ENERGY) {
                e += a.fc.eps4 * s6 * (s6 - 1.0) - a.fc.shift;
                ++npair;
            }
        });
    }
    if (ENERGY) {
        e = lanes_sum<P>(e);
        if (on) count_pairs(a.ds, npair);
        if (on && part == 0) a.e_atom[i] = 0.5 * e;
    }
    f64_finish<MODE, false, P>(a, i, part, on, fx, fy, fz, qw, store_f);
}

// One thread per sorted atom; the hardware block scheduler spreads the work.
// Block shape of the grid kernel, measured on GB300: 128 threads for one
// box and 256 for batches, each at up to 56 registers (4-9 % faster than
// 256 threads at 48 registers).
template <bool MULTI>
constexpr int grid_block() { return MULTI ? 256 : 128; }

// P > 1: thread t serves atom t / P (blocks of 128).
template <int MODE, bool ENERGY, bool MULTI = false, int P = 1>
__global__ void __launch_bounds__(P > 1 ? 128 : grid_block<MULTI>(), P > 1 ? 1 : (MULTI ? 4 : 5))
lj_mixed_kernel(ForceArgs a, int store_f) {
    if (a.ds->status != 0) return;
    step_bookkeeping<MODE>(a);
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if constexpr (P > 1) {
        const bool on = t / P < a.n;
        lj_mixed_atom<MODE, ENERGY, MULTI, P>(a, on ? t / P : a.n - 1, store_f, t % P, on);
    } else if (t < a.n) {
        lj_mixed_atom<MODE, ENERGY, MULTI>(a, t, store_f);
    }
}

// Persistent variant: gridDim.x CTAs stay resident; each warp processes tiles
// of 32 consecutive sorted atoms (tile t = atoms 32t .. 32t+31, aligned with
// the list layout).
//   STATIC:  the cells are cut into rounds * G contiguous ranges of equal
//            (predicted) cost; CTA b owns ranges b, b + G, b + 2G, ... and its
//            warps claim their tiles from a shared counter.  A range starts at
//            the first whole tile of its first cell, so no tile is split
//            between two ranges (and no lane idles at a range boundary).  Each CTA gets the
//            same predicted total, while at any moment all CTAs work in the
//            same window of the sorted atoms, which keeps neighbour gathers
//            in L2.
//            The cells after the static ranges (the partition's last parts,
//            a fifth of the predicted cost) form a tail that warps
//            claim from a global counter, one tile at a time, once their
//            CTA's ranges are done: whichever CTA is early absorbs the error
//            of the prediction.
//   DYNAMIC: warps claim tiles from a global counter until none are left.
//   Either way the last CTA to finish resets the counter for the next launch.
// TIMING adds clock64 per tile: the tile's cycles are shared equally by its
// active atoms and added to their cells (cell_cycles), and each CTA's busy
// cycles go to cta_cycles -- the training data of the cost model.
constexpr int kClaim = 8;      // tiles claimed per atomic by the dynamic queue
constexpr int kClaimTail = 1;  // tiles claimed per atomic from the static mode's tail

__device__ __forceinline__ void prefetch_l2(const void *p) {
    asm volatile("prefetch.global.L2 [%0];" ::"l"(p));
}

// F64: the same scheduling of the plain float64 per-atom job (the baseline
// the mixed path is measured against).  PAIRED: the items are the two-atom
// slots of MD_FORCE_PAIRED (tiles of 32 slots; sa.cell_start then holds the
// first slot of every cell) and each runs the slot job of k_pair.cuh.
// CTAs of 128 threads at up to 56 registers (9 per SM) were measured fastest:
// 1.359 ms against 1.395 ms for 256 threads at 48 registers on the 9.8 M-atom
// porous system.
constexpr int kPersistBlock = kPersistThreads;
static_assert(kPersistBlock == kF64Block, "the float64 job's shared columns");
// The slot job fits 56 registers too.
constexpr int kPersistPairedCtas = 9;

template <int MODE, bool ENERGY, bool DYNAMIC, bool TIMING, bool MULTI = false, bool F64 = false,
          bool PAIRED = false>
__global__ void __launch_bounds__(kPersistBlock, F64 ? 8 : (PAIRED ? kPersistPairedCtas : 9))
lj_mixed_persist(ForceArgs a, int store_f, SchedArgs sa, PairArgs pa) {

    static_assert(!(F64 && MULTI), "batches run the mixed path");
    static_assert(!(PAIRED && (F64 || MULTI || ENERGY)), "slots: one box, mixed path, forces");
    // Per-atom tiles of one box read the cell shifts from a table here: computed
    // ones made the launch 6-8 % shorter (2.1 M porous atoms: 319 -> 293 us) but the
    // tiles' timings, which train the cost model, noisier: the model's held-out
    // spread over 64 parts went from 0.0215-0.0225 to 0.0224-0.0269, no longer
    // surely below the pair count's.
    constexpr bool kTable = F64 || !(MULTI || PAIRED);
    __shared__ typename std::conditional<kTable, ShiftTab, int>::type sh;
    __shared__ typename std::conditional<F64, Home64, int>::type home;
    __shared__ int s_first[kSchedRounds], s_pre[kSchedRounds + 1], s_next;  // this CTA's ranges
    __shared__ int s_stop;
    if constexpr (kTable) load_shifts_f32(a.g, &sh);
    // one read of the status word for the whole CTA: every thread must take the
    // same branch, since the CTA meets barriers below
    if (threadIdx.x == 0) s_stop = a.ds->status;
    __syncthreads();
    if (s_stop != 0) return;
    step_bookkeeping<MODE>(a);
    const int lane = threadIdx.x & 31;
    const int nitems = PAIRED ? pa.slot_start[pa.ncells] : a.n;
    const int ntiles = (nitems + 31) >> 5;
    long long cta_t0 = 0;
    if (TIMING) cta_t0 = clock64();
    // The claim state lives in shared memory (the CTA's ranges, and each
    // warp's queue cursor), so that no register is held through the work of
    // a tile: the slot job needs all of them.
    __shared__ int s_nlocal, s_tail0;
    __shared__ int s_wq[kPersistBlock / 32][4];  // per warp: claim end, next, range, local done
    if (threadIdx.x == 0) {
        s_nlocal = 0;
        s_tail0 = ntiles;
    }
    if (lane < 4) s_wq[threadIdx.x >> 5][lane] = (lane == 3) ? (DYNAMIC ? 1 : 0) : 0;
    if (!DYNAMIC) {
        // cyclic static partition: this CTA owns ranges b, b + G, b + 2G, ...
        // so that at any time all CTAs work in one window of the sorted atoms
        // (neighbour gathers then hit in L2).  Its warps claim the ranges'
        // tiles one at a time from a shared counter, so they finish together.
        if (threadIdx.x == 0) {
            const long long qt = (long long)sa.rounds * gridDim.x;
            s_tail0 = (sa.cell_start[sa.bounds[qt]] + 31) >> 5;
            int acc = 0;
            for (int r = 0; r < sa.rounds; ++r) {
                const long long q = (long long)r * gridDim.x + blockIdx.x;
                const int tf = (sa.cell_start[sa.bounds[q]] + 31) >> 5;
                const int te = (sa.cell_start[sa.bounds[q + 1]] + 31) >> 5;
                s_first[r] = tf;
                s_pre[r] = acc;
                acc += te - tf;
            }
            s_pre[sa.rounds] = acc;
            s_nlocal = acc;
            s_next = 0;
        }
    }
    __syncthreads();
    // next tile of this warp, or -1 when none is left; every lane computes the
    // same values, so the lanes' identical stores to the warp's cursor agree
    auto claim = [&]() -> int {
        int *wq = s_wq[threadIdx.x >> 5];
        int res = -1;
        bool done = wq[3] != 0;
        if (!done) {
            int k = 0;
            if (lane == 0) k = atomicAdd(&s_next, 1);
            k = __shfl_sync(0xffffffffu, k, 0);
            if (k < s_nlocal) {
                int r = wq[2];  // this warp's claims only grow: its range only advances
                while (k >= s_pre[r + 1]) ++r;
                res = s_first[r] + (k - s_pre[r]);
                __syncwarp();
                wq[2] = r;
            } else {
                done = true;
                __syncwarp();
                wq[3] = 1;
            }
        }
        if (done) {
            // the global queue: all tiles (dynamic mode) or the tail (static mode)
            const int base = DYNAMIC ? 0 : s_tail0;
            const int step = DYNAMIC ? kClaim : kClaimTail;
            int tnext = wq[1], cend = wq[0];
            if (tnext >= cend) {
                int c = 0;
                if (lane == 0) c = atomicAdd(&a.ds->tile_counter, step);
                tnext = base + __shfl_sync(0xffffffffu, c, 0);
                cend = tnext + step;
            }
            if (tnext < ntiles) res = tnext++;
            __syncwarp();
            wq[1] = tnext;
            wq[0] = cend;
        }
        __syncwarp();
        return res;
    };
    int t = claim();
    while (t >= 0) {
        // claim the next tile now and bring its list head, position and count
        // into L2 while this tile runs (a grid launch gets this overlap from
        // its next CTAs)
        const int tn = claim();
        if (tn >= 0) {
            const int in = (tn << 5) + lane;
            if (in < nitems) {
                if (PAIRED) {
                    prefetch_l2(pa.list + list_group(in, pa.cap) + ((in & 31) << 2));
                    prefetch_l2(pa.slot_atom + in);
                    prefetch_l2(pa.count + in);
                } else {
                    prefetch_l2(a.nlist + list_group(in, a.cap) + ((in & 31) << 2));
                    if (F64) prefetch_l2(a.xr + in);
                    else prefetch_l2(a.xq + in);
                    prefetch_l2(a.ncount + in);
                }
            }
        }
        const int i = (t << 5) + lane;
        const bool active = i < nitems;
        long long t0 = 0;
        if (TIMING) {
            __syncwarp();
            t0 = clock64();
        }
        if constexpr (F64) {
            lj_fp64_atom<MODE, ENERGY, 1>(a, &sh, &home, active ? i : 0, 0, active, store_f);
        } else if (active) {
            if constexpr (PAIRED) lj_pair_slot<MODE, false>(a, pa, i, store_f);
            else if constexpr (MULTI) lj_mixed_atom<MODE, ENERGY, true>(a, i, store_f);
            else lj_mixed_atom<MODE, ENERGY, false, 1, true>(a, i, store_f, 0, true, &sh);
        }
        if (TIMING) {
            __syncwarp();
            const long long dt = clock64() - t0;
            const unsigned act = __ballot_sync(0xffffffffu, active);
            if (active) {
                const int c = PAIRED ? sa.cell[pa.slot_atom[i] & ~kSingle] : sa.cell[i];
                atomicAdd(&sa.cell_cycles[c], (float)dt / (float)__popc(act));
            }
        }
        t = tn;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        if (TIMING) sa.cta_cycles[blockIdx.x] += (float)(clock64() - cta_t0);
        {
            __threadfence();
            const unsigned prev = atomicAdd(&a.ds->done_ctas, 1u);
            if (prev == gridDim.x - 1) {
                a.ds->tile_counter = 0;
                a.ds->done_ctas = 0;
                __threadfence();
            }
        }
    }
}

template <int MODE, bool ENERGY, int P>
__global__ void __launch_bounds__(kF64Block) lj_fp64_kernel(ForceArgs a, int store_f) {
    __shared__ ShiftTab sh;
    __shared__ Home64 home;
    load_shifts_f32(a.g, &sh);
    __syncthreads();
    if (a.ds->status != 0) return;
    step_bookkeeping<MODE>(a);
    const long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    const bool on = t < (long long)a.n * P;
    lj_fp64_atom<MODE, ENERGY, P>(a, &sh, &home, on ? (int)(t / P) : 0, (int)(t % P), on, store_f);
}

template <int P>
cudaError_t launch_lj_fp64(const ForceArgs &a, int mode, bool energy, int sf, cudaStream_t s) {
    const int nb = nblocks((int64_t)a.n * P, kF64Block);
    switch (mode) {
        case FM_STORE:
            if (energy) lj_fp64_kernel<FM_STORE, true, P><<<nb, kF64Block, 0, s>>>(a, sf);
            else lj_fp64_kernel<FM_STORE, false, P><<<nb, kF64Block, 0, s>>>(a, sf);
            break;
        case FM_FUSED_FULL: lj_fp64_kernel<FM_FUSED_FULL, false, P><<<nb, kF64Block, 0, s>>>(a, sf); break;
        default: lj_fp64_kernel<FM_FUSED_HALF, false, P><<<nb, kF64Block, 0, s>>>(a, sf); break;
    }
    return cudaGetLastError();
}

// ---- multi-element Lennard-Jones (Sec. 2.2 pair loop, Sec. 3.1 Cu-Au) ------
//
// The paper's SIMD loop reloads the parameters of each pair with masks.  Here
// the lane keeps the row of its own species (NT values of each parameter) in
// registers and picks the pair's entry with the species of j, which sits in
// the position word it loads anyway: selects instead of loads.

template <int NT>
__device__ __forceinline__ float pick_row(const float *row, int t) {
    if (NT == 1) return row[0];
    if (NT == 2) return t ? row[1] : row[0];
    if (NT == 3) return t == 0 ? row[0] : (t == 1 ? row[1] : row[2]);
    return t < 2 ? (t == 0 ? row[0] : row[1]) : (t == 2 ? row[2] : row[3]);
}
template <int NT>
__device__ __forceinline__ double pick_row(const double *row, int t) {
    if (NT == 1) return row[0];
    if (NT == 2) return t ? row[1] : row[0];
    if (NT == 3) return t == 0 ? row[0] : (t == 1 ? row[1] : row[2]);
    return t < 2 ? (t == 0 ? row[0] : row[1]) : (t == 2 ? row[2] : row[3]);
}
// row ti of an NT x NT table, into registers (constant indices only)
template <int NT, class T>
__device__ __forceinline__ void load_row(const T *tab, int ti, T *row) {
#pragma unroll
    for (int k = 0; k < NT; ++k) {
        T v = tab[k];
#pragma unroll
        for (int r = 1; r < NT; ++r) v = (ti == r) ? tab[r * NT + k] : v;
        row[k] = v;
    }
}

template <int MODE, bool ENERGY, int NT, int P>
__device__ __forceinline__ void lj_typed_mixed_atom(const ForceArgs &a, const TypeTab &tt,
                                                    int i, int store_f, int part, bool on) {
    const float4 qi = a.xq[i];
    const int ti = species_of(__float_as_uint(qi.w));
    float e48[NT], e4[NT], s2[NT], shf[NT];
    load_row<NT>(tt.e48, ti, e48);
    load_row<NT>(tt.e4, ti, e4);
    load_row<NT>(tt.s2, ti, s2);
    load_row<NT>(tt.sh, ti, shf);
    const int nq = (min(a.ncount[i], a.cap) + 3) >> 2;
    const uint4 *lq = reinterpret_cast<const uint4 *>(a.nlist + list_group(i, a.cap)) + (i & 31);
    const float rc2 = a.fc.rc2f;
    double Fx = 0.0, Fy = 0.0, Fz = 0.0, E = 0.0;
    unsigned npair = 0;
    float fx = 0.f, fy = 0.f, fz = 0.f, e = 0.f;
    auto pair = [&](uint32_t ent) {
        const float4 qj = __ldg(a.xq + (ent & kIndexMask));
        const float3 st = stencil_of(ent);
        const float ex = fmaf(st.x, a.g.wf[0], qj.x - qi.x);
        const float ey = fmaf(st.y, a.g.wf[1], qj.y - qi.y);
        const float ez = fmaf(st.z, a.g.wf[2], qj.z - qi.z);
        const float r2 = dist2(ex, ey, ez);
        if (r2 < rc2) {
            const int tj = species_of(__float_as_uint(qj.w));
            const float r2i = rcp_fast(r2);
            float s6 = pick_row<NT>(s2, tj) * r2i;
            s6 = s6 * s6 * s6;
            const float fs = pick_row<NT>(e48, tj) * r2i * s6 * (s6 - 0.5f);
            fx -= fs * ex;
            fy -= fs * ey;
            fz -= fs * ez;
            if (ENERGY) {
                e += pick_row<NT>(e4, tj) * s6 * (s6 - 1.0f) - pick_row<NT>(shf, tj);
                ++npair;
            }
        }
    };
    if constexpr (P > 1) {
        const int c = part & 3;
        const SplitState t = load_split_state<MODE>(a, i, c, on && part < 4);
        split_quads<P>(lq, on ? nq : 0, part, pair);
        const double F = split_component<P>(fx, fy, fz, e, part);
        if (ENERGY) {
            if (on) count_pairs(a.ds, npair);
            if (on && part == 3) a.e_atom[i] = 0.5 * F;
        }
        split_epilogue<MODE, true>(a, i, c, on && part < 4, F, qi.w, t, store_f);
        return;
    }
    uint4 nxt = nq > 0 ? __ldcs(lq) : make_uint4(0u, 0u, 0u, 0u);
    for (int q0 = 0; q0 < nq; q0 += kChunkQ) {
        const int q1 = min(q0 + kChunkQ, nq);
        for (int q = q0; q < q1; ++q) {
            const uint4 e4q = nxt;
            if (q + 1 < nq) nxt = __ldcs(lq + (size_t)(q + 1) * 32);
            pair(e4q.x);
            pair(e4q.y);
            pair(e4q.z);
            pair(e4q.w);
        }
        Fx += (double)fx;
        Fy += (double)fy;
        Fz += (double)fz;
        fx = fy = fz = 0.f;
        if (ENERGY) {
            E += (double)e;
            e = 0.f;
        }
    }
    const size_t n = (size_t)a.n;
    if (MODE == FM_STORE || store_f) {
        a.f[i] = Fx;
        a.f[n + i] = Fy;
        a.f[2 * n + i] = Fz;
    }
    if (ENERGY) {
        a.e_atom[i] = 0.5 * E;
        count_pairs(a.ds, npair);
    }
    if (MODE != FM_STORE) vv_epilogue<MODE, true>(a, i, Fx, Fy, Fz, qi.w);
}

template <int MODE, bool ENERGY, int NT, int P>
__device__ __forceinline__ void lj_typed_fp64_atom(const ForceArgs &a, const TypeTab &tt,
                                                   const ShiftTab *sh, Home64 *h, int i, int part,
                                                   bool on, int store_f) {
    double fx = 0.0, fy = 0.0, fz = 0.0, e = 0.0;
    unsigned npair = 0;
    float qw = 0.f;
    load_home64<P>(a, i, part, h);
    if (on) {
        const float4 qi = a.xq[i];
        qw = qi.w;
        const int ti = species_of(__float_as_uint(qi.w));
        double e48[NT], e4[NT], s2[NT], shd[NT];
        load_row<NT>(tt.e48d, ti, e48);
        load_row<NT>(tt.e4d, ti, e4);
        load_row<NT>(tt.s2d, ti, s2);
        load_row<NT>(tt.shd, ti, shd);
        const int seed_hi = a.fc.f64_seed_hi;
        f64_pairs<P>(a, sh, h, i, part, qi, [&](int j, double ex, double ey, double ez, double r2) {
            const int tj = species_of(__float_as_uint(__ldg(&a.xq[j].w)));
            const double r2i = rcp_f64(r2, seed_hi);
            double s6 = pick_row<NT>(s2, tj) * r2i;
            s6 = s6 * s6 * s6;
            const double fs = (pick_row<NT>(e48, tj) * r2i) * fma(s6, s6, -0.5 * s6);
            fx -= fs * ex;
            fy -= fs * ey;
            fz -= fs * ez;
            if (ENERGY) {
                e += pick_row<NT>(e4, tj) * s6 * (s6 - 1.0) - pick_row<NT>(shd, tj);
                ++npair;
            }
        });
    }
    if (ENERGY) {
        e = lanes_sum<P>(e);
        if (on) count_pairs(a.ds, npair);
        if (on && part == 0) a.e_atom[i] = 0.5 * e;
    }
    f64_finish<MODE, true, P>(a, i, part, on, fx, fy, fz, qw, store_f);
}

template <int MODE, bool ENERGY, int NT, int P>
__global__ void __launch_bounds__(kF64Block) lj_typed_fp64_kernel(ForceArgs a, TypeTab tt,
                                                                  int store_f) {
    __shared__ ShiftTab sh;
    __shared__ Home64 home;
    load_shifts_f32(a.g, &sh);
    __syncthreads();
    if (a.ds->status != 0) return;
    step_bookkeeping<MODE>(a);
    const long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    const bool on = t < (long long)a.n * P;
    lj_typed_fp64_atom<MODE, ENERGY, NT, P>(a, tt, &sh, &home, on ? (int)(t / P) : 0, (int)(t % P),
                                            on, store_f);
}

template <int MODE, bool ENERGY, int NT, int P>
__global__ void __launch_bounds__(128) lj_typed_kernel(ForceArgs a, TypeTab tt, int store_f) {
    if (a.ds->status != 0) return;
    step_bookkeeping<MODE>(a);
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    const bool on = t / P < a.n;
    if (P == 1 && !on) return;
    lj_typed_mixed_atom<MODE, ENERGY, NT, P>(a, tt, on ? t / P : a.n - 1, store_f, t % P, on);
}

template <int NT, int P>
cudaError_t launch_lj_typed_mixed(md_system *h, const ForceArgs &a, int mode, bool energy, int sf) {
    const int nb = nblocks((int64_t)a.n * P, 128);
    cudaStream_t s = h->stream;
    const TypeTab &tt = h->types;
    switch (mode) {
        case FM_STORE:
            if (energy) lj_typed_kernel<FM_STORE, true, NT, P><<<nb, 128, 0, s>>>(a, tt, sf);
            else lj_typed_kernel<FM_STORE, false, NT, P><<<nb, 128, 0, s>>>(a, tt, sf);
            break;
        case FM_FUSED_FULL:
            lj_typed_kernel<FM_FUSED_FULL, false, NT, P><<<nb, 128, 0, s>>>(a, tt, sf);
            break;
        default: lj_typed_kernel<FM_FUSED_HALF, false, NT, P><<<nb, 128, 0, s>>>(a, tt, sf); break;
    }
    return cudaGetLastError();
}

template <int NT, int P>
cudaError_t launch_lj_typed_fp64(md_system *h, const ForceArgs &a, int mode, bool energy, int sf) {
    const int nb = nblocks((int64_t)a.n * P, kF64Block);
    cudaStream_t s = h->stream;
    const TypeTab &tt = h->types;
    switch (mode) {
        case FM_STORE:
            if (energy) lj_typed_fp64_kernel<FM_STORE, true, NT, P><<<nb, kF64Block, 0, s>>>(a, tt, sf);
            else lj_typed_fp64_kernel<FM_STORE, false, NT, P><<<nb, kF64Block, 0, s>>>(a, tt, sf);
            break;
        case FM_FUSED_FULL:
            lj_typed_fp64_kernel<FM_FUSED_FULL, false, NT, P><<<nb, kF64Block, 0, s>>>(a, tt, sf);
            break;
        default:
            lj_typed_fp64_kernel<FM_FUSED_HALF, false, NT, P><<<nb, kF64Block, 0, s>>>(a, tt, sf);
            break;
    }
    return cudaGetLastError();
}

template <int NT>
cudaError_t launch_lj_typed_nt(md_system *h, const ForceArgs &a, int mode, bool energy, int sf) {
    if (h->p.precision == MD_MIXED)
        return split8(h->n, h->cap, kTypedSplit) > 1 ? launch_lj_typed_mixed<NT, 8>(h, a, mode, energy, sf)
                                             : launch_lj_typed_mixed<NT, 1>(h, a, mode, energy, sf);
    switch (f64_split(h->n)) {
        case 1: return launch_lj_typed_fp64<NT, 1>(h, a, mode, energy, sf);
        case 4: return launch_lj_typed_fp64<NT, 4>(h, a, mode, energy, sf);
        case 8: return launch_lj_typed_fp64<NT, 8>(h, a, mode, energy, sf);
        default: return launch_lj_typed_fp64<NT, 16>(h, a, mode, energy, sf);
    }
}

cudaError_t launch_lj_typed(md_system *h, const ForceArgs &a, int mode, bool energy, int sf) {
    switch (h->fc.ntypes) {
        case 1: return launch_lj_typed_nt<1>(h, a, mode, energy, sf);
        case 2: return launch_lj_typed_nt<2>(h, a, mode, energy, sf);
        case 3: return launch_lj_typed_nt<3>(h, a, mode, energy, sf);
        default: return launch_lj_typed_nt<4>(h, a, mode, energy, sf);
    }
}

ForceArgs make_force_args(md_system *h) {
    ForceArgs a;
    a.n = (int)h->n;
    a.cap = h->cap;
    a.step = (int)h->steps_total;
    a.rebuild_every = h->p.rebuild_every;
    int cur = h->cur, nxt = cur ^ 1;
    a.xq = h->xq[cur];
    a.xq_out = h->xq[nxt];
    a.xr = h->xr64[cur];
    a.xr_out = h->xr64[nxt];
    a.xq_build = h->xq_build;
    a.v = h->v;
    a.f = h->f;
    a.e_atom = h->e_atom;
    a.nlist = h->nlist;
    a.ncount = h->ncount;
    a.rho = h->rho;
    a.dF32 = h->dF32;
    a.xqf = h->xqf;
    a.dF64 = h->dF64;
    a.rep = h->rep;
    a.widths32 = h->widths32;
    a.ds = h->ds;
    a.g = h->g;
    a.fc = h->fc;
    return a;
}

template <bool MULTI, int P>
cudaError_t launch_lj_mixed(const ForceArgs &a, int mode, bool energy, int sf, cudaStream_t s) {
    const int tb = P > 1 ? 128 : grid_block<MULTI>();
    const int nb = nblocks((int64_t)a.n * P, tb);
    switch (mode) {
        case FM_STORE:
            if (energy) lj_mixed_kernel<FM_STORE, true, MULTI, P><<<nb, tb, 0, s>>>(a, sf);
            else lj_mixed_kernel<FM_STORE, false, MULTI, P><<<nb, tb, 0, s>>>(a, sf);
            break;
        case FM_FUSED_FULL: lj_mixed_kernel<FM_FUSED_FULL, false, MULTI, P><<<nb, tb, 0, s>>>(a, sf); break;
        default: lj_mixed_kernel<FM_FUSED_HALF, false, MULTI, P><<<nb, tb, 0, s>>>(a, sf); break;
    }
    return cudaGetLastError();
}

cudaError_t launch_lj(md_system *h, int mode, bool energy, bool store_f) {
    ForceArgs a = make_force_args(h);
    const int sf = store_f ? 1 : 0;
    cudaStream_t s = h->stream;
    if (h->fc.ntypes > 0) return launch_lj_typed(h, a, mode, energy, sf);
    if (h->p.precision == MD_MIXED) {
        const int P = mixed_split(h->n, h->cap, kFourLanesAtoms);
        if (h->R > 1)
            return P == 8 ? launch_lj_mixed<true, 8>(a, mode, energy, sf, s)
                 : P == 4 ? launch_lj_mixed<true, 4>(a, mode, energy, sf, s)
                          : launch_lj_mixed<true, 1>(a, mode, energy, sf, s);
        return P == 8 ? launch_lj_mixed<false, 8>(a, mode, energy, sf, s)
             : P == 4 ? launch_lj_mixed<false, 4>(a, mode, energy, sf, s)
                      : launch_lj_mixed<false, 1>(a, mode, energy, sf, s);
    } else {
        switch (f64_split(h->n)) {
            case 1: return launch_lj_fp64<1>(a, mode, energy, sf, s);
            case 4: return launch_lj_fp64<4>(a, mode, energy, sf, s);
            case 8: return launch_lj_fp64<8>(a, mode, energy, sf, s);
            default: return launch_lj_fp64<16>(a, mode, energy, sf, s);
        }
    }
    return cudaGetLastError();
}

}  // namespace mdg

namespace mdg {

int persist_ctas_per_sm(bool f64, bool paired) {
    int nb = 0;
    const cudaError_t e =
        f64 ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(
                  &nb, lj_mixed_persist<FM_FUSED_FULL, false, false, false, false, true>, kPersistBlock, 0)
        : paired ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(
                  &nb, lj_mixed_persist<FM_FUSED_FULL, false, false, false, false, false, true>,
                  kPersistBlock, 0)
            : cudaOccupancyMaxActiveBlocksPerMultiprocessor(
                  &nb, lj_mixed_persist<FM_FUSED_FULL, false, false, false>, kPersistBlock, 0);
    if (e != cudaSuccess) nb = 1;
    return nb > 0 ? nb : 1;
}

cudaError_t launch_lj_persist(md_system *h, int mode, bool store_f, bool dynamic, bool timing) {
    ForceArgs a = make_force_args(h);
    const bool paired = (h->p.force_variant == MD_FORCE_PAIRED);
    SchedArgs sa;
    sa.cell_start = paired ? h->ps_start : h->cell_start;
    sa.bounds = h->part_bounds;
    sa.cell = h->cell;
    sa.cell_cycles = h->cell_cycles;
    sa.cta_cycles = h->cta_cycles;
    sa.rounds = h->sched_rounds;
    const PairArgs pa = paired ? make_pair_args(h) : PairArgs{};
    const int G = h->sched_ctas;
    const int sf = store_f ? 1 : 0;
    cudaStream_t s = h->stream;
    if (h->R > 1) {
        // several boxes: the tile queue (the static partitions are single-box)
        switch (mode) {
            case FM_STORE:
                lj_mixed_persist<FM_STORE, false, true, false, true><<<G, kPersistBlock, 0, s>>>(a, sf, sa, pa);
                break;
            case FM_FUSED_FULL:
                lj_mixed_persist<FM_FUSED_FULL, false, true, false, true><<<G, kPersistBlock, 0, s>>>(a, sf, sa, pa);
                break;
            default:
                lj_mixed_persist<FM_FUSED_HALF, false, true, false, true><<<G, kPersistBlock, 0, s>>>(a, sf, sa, pa);
                break;
        }
        return cudaGetLastError();
    }
    if (timing) {
        if (paired) {
            if (dynamic) lj_mixed_persist<FM_STORE, false, true, true, false, false, true><<<G, kPersistBlock, 0, s>>>(a, 1, sa, pa);
            else lj_mixed_persist<FM_STORE, false, false, true, false, false, true><<<G, kPersistBlock, 0, s>>>(a, 1, sa, pa);
        } else {
            if (dynamic) lj_mixed_persist<FM_STORE, false, true, true><<<G, kPersistBlock, 0, s>>>(a, 1, sa, pa);
            else lj_mixed_persist<FM_STORE, false, false, true><<<G, kPersistBlock, 0, s>>>(a, 1, sa, pa);
        }
        return cudaGetLastError();
    }
    const bool f64 = (h->p.precision == MD_FP64);
#define MDG_P(M)                                                                               \
    do {                                                                                       \
        if (paired) {                                                                          \
            if (dynamic)                                                                       \
                lj_mixed_persist<M, false, true, false, false, false, true><<<G, kPersistBlock, 0, s>>>(a, sf, sa, pa);  \
            else                                                                               \
                lj_mixed_persist<M, false, false, false, false, false, true><<<G, kPersistBlock, 0, s>>>(a, sf, sa, pa); \
        } else if (f64) {                                                                      \
            if (dynamic)                                                                       \
                lj_mixed_persist<M, false, true, false, false, true><<<G, kPersistBlock, 0, s>>>(a, sf, sa, pa);  \
            else                                                                               \
                lj_mixed_persist<M, false, false, false, false, true><<<G, kPersistBlock, 0, s>>>(a, sf, sa, pa); \
        } else if (dynamic) {                                                                  \
            lj_mixed_persist<M, false, true, false><<<G, kPersistBlock, 0, s>>>(a, sf, sa, pa);            \
        } else {                                                                               \
            lj_mixed_persist<M, false, false, false><<<G, kPersistBlock, 0, s>>>(a, sf, sa, pa);           \
        }                                                                                      \
    } while (0)
    switch (mode) {
        case FM_STORE: MDG_P(FM_STORE); break;
        case FM_FUSED_FULL: MDG_P(FM_FUSED_FULL); break;
        default: MDG_P(FM_FUSED_HALF); break;
    }
#undef MDG_P
    return cudaGetLastError();
}

}  // namespace mdg
