// k_pair.cuh -- the per-slot job of the two-atoms-per-thread force pass
// (MD_FORCE_PAIRED), shared by its grid kernel (k_pair.cu) and the
// persistent kernel of the schedulers (k_lj.cu).  The layout, the list and
// the arithmetic are described at the top of k_pair.cu.
#pragma once

#include "k_common.cuh"
#include "k_packed.cuh"

namespace mdg {

constexpr uint32_t kSingle = 0x80000000u;  // slot_atom: a one-atom slot

struct PairArgs {
    const int32_t *slot_start;   // ncells + 1 (slot_start[ncells] = slots)
    const uint32_t *slot_atom;
    const uint32_t *list;
    const int32_t *count;
    int cap, ncells;
};

// The slot tables and union lists of a handle, for the kernels.
inline PairArgs make_pair_args(const md_system *h) {
    PairArgs p;
    p.slot_start = h->ps_start;
    p.slot_atom = h->ps_atom;
    p.list = h->ps_list;
    p.count = h->ps_count;
    p.cap = h->ps_cap;
    p.ncells = h->g.ncells;
    return p;
}

// Blocks of `block` threads that cover every slot a binning can make, P lanes
// per slot.
inline int pair_grid_blocks(const md_system *h, int block, int P = 1) {
    return (int)((pair_slots_max(h->n, h->g.ncells) * P + block - 1) / block);
}

// Lennard-Jones pair term in float32 for the pair vector e = x_j - x_i:
// f_i -= fs * e; with ENERGY the shifted pair energy is added to `en`.
template <bool ENERGY>
__device__ __forceinline__ void lj_term(const ForceConsts &fc, float ex, float ey, float ez,
                                        float r2, float &fx, float &fy, float &fz, float &en,
                                        unsigned &np) {
    const float r2i = rcp_fast(r2);
    float s6 = fc.sig2f * r2i;
    s6 = s6 * s6 * s6;
    const float fs = fc.eps48f * r2i * s6 * (s6 - 0.5f);
    fx -= fs * ex;
    fy -= fs * ey;
    fz -= fs * ez;
    if (ENERGY) {
        en += fc.eps4f * s6 * (s6 - 1.0f) - fc.shiftf;
        ++np;
    }
}

// Stores, energies and the velocity-Verlet epilogue of one atom of a slot.
template <int MODE, bool ENERGY>
__device__ __forceinline__ void pair_atom_out(const ForceArgs &a, int i, double Fx, double Fy,
                                              double Fz, double E, unsigned np, float qw,
                                              int store_f) {
    const size_t n = (size_t)a.n;
    if (MODE == FM_STORE || store_f) {
        a.f[i] = Fx;
        a.f[n + i] = Fy;
        a.f[2 * n + i] = Fz;
    }
    if (ENERGY) {
        a.e_atom[i] = 0.5 * E;
        count_pairs(a.ds, np);
    }
    if (MODE != FM_STORE) vv_epilogue<MODE>(a, i, Fx, Fy, Fz, qw);
}

// State of the components that the lane finishes: with eight lanes component
// part % 4 of atom part / 4, with four that of both atoms.
template <int MODE, int P>
__device__ __forceinline__ void load_slot_state(const ForceArgs &a, int i0, bool two, bool on,
                                                int part, SplitState &t, SplitState &t1) {
    const int c = part & 3, k = P >= 8 ? (part >> 2) & 1 : 0;
    t = load_split_state<MODE>(a, i0 + (two ? k : 0), c, on && part < 8);
    t1 = P < 8 ? load_split_state<MODE>(a, i0 + (two ? 1 : 0), c, on) : t;
}

// Stores and epilogues of a slot's atoms from their forces, which every one of its
// P lanes holds (every lane of the warp calls it).
template <int MODE, bool SPECIES, int P>
__device__ __forceinline__ void split_slot_finish(const ForceArgs &a, int i0, bool two, bool on,
                                                  int part, const double *F0, const double *F1,
                                                  const SplitState &t, const SplitState &t1,
                                                  int store_f) {
    const int c = part & 3;
    const double G0 = c == 0 ? F0[0] : (c == 1 ? F0[1] : F0[2]);
    const double G1 = c == 0 ? F1[0] : (c == 1 ? F1[1] : F1[2]);
    const float *words = reinterpret_cast<const float *>(a.xq);
    const int i1 = i0 + (two ? 1 : 0);
    if (P >= 8) {
        const bool second = (part >> 2) & 1;
        const int i = second ? i1 : i0;
        split_epilogue<MODE, SPECIES>(a, i, c, on && part < 8 && (two || !second), second ? G1 : G0,
                                      words[4 * (size_t)i + 3], t, store_f);
    } else {
        split_epilogue<MODE, SPECIES>(a, i0, c, on, G0, words[4 * (size_t)i0 + 3], t, store_f);
        split_epilogue<MODE, SPECIES>(a, i1, c, on && two, G1, words[4 * (size_t)i1 + 3], t1, store_f);
    }
}

// Sums of a slot's P lanes, then stores, energies and epilogues of its atoms (every
// lane of the warp calls it): t is the state of the lane's component of the first
// atom (with eight lanes: of atom part / 4), t1 that of the second with four.
template <int MODE, bool ENERGY, bool SPECIES, int P>
__device__ __forceinline__ void split_slot_out(const ForceArgs &a, int i0, bool two, bool on,
                                               int part, float2 fx, float2 fy, float2 fz,
                                               float2 en, unsigned np0, unsigned np1,
                                               const SplitState &t, const SplitState &t1,
                                               int store_f) {
    fx = make_float2(split_sum<P>(fx.x), split_sum<P>(fx.y));
    fy = make_float2(split_sum<P>(fy.x), split_sum<P>(fy.y));
    fz = make_float2(split_sum<P>(fz.x), split_sum<P>(fz.y));
    if (ENERGY) {
        en = make_float2(split_sum<P>(en.x), split_sum<P>(en.y));
        if (on) count_pairs(a.ds, np0 + (two ? np1 : 0u));
        if (on && part == 0) a.e_atom[i0] = 0.5 * (double)en.x;
        if (on && two && part == 1) a.e_atom[i0 + 1] = 0.5 * (double)en.y;
    }
    const double F0[3] = {(double)fx.x, (double)fy.x, (double)fz.x};
    const double F1[3] = {(double)fx.y, (double)fy.y, (double)fz.y};
    split_slot_finish<MODE, SPECIES, P>(a, i0, two, on, part, F0, F1, t, t1, store_f);
}

// MULTI (a batch of boxes): the cell widths are those of the slot's box.
// P > 1: the P lanes of the slot (this one is `part`; on: the slot exists) each
// walk every P-th quad of its list; lane 0 adds the slot's own pair.
template <int MODE, bool ENERGY, bool MULTI = false, int P = 1>
__device__ __forceinline__ void lj_pair_slot(const ForceArgs &a, const PairArgs &p, int s,
                                             int store_f, int part = 0, bool on = true) {
    const uint32_t sa = p.slot_atom[s];
    const int i0 = (int)(sa & ~kSingle);
    const float3 w = MULTI ? replica_width(a, (int)a.rep[i0])
                           : make_float3(a.g.wf[0], a.g.wf[1], a.g.wf[2]);
    const bool two = !(sa & kSingle);
    const float4 q0 = a.xq[i0];
    // a one-atom slot puts its second atom at the dummy's distance
    const float4 q1 = two ? a.xq[i0 + 1] : make_float4(3.0e18f, 3.0e18f, 3.0e18f, 0.f);
    const float rc2 = a.fc.rc2f;
    float2 fx = dup2(0.f), fy = dup2(0.f), fz = dup2(0.f), en = dup2(0.f);
    unsigned np0 = 0, np1 = 0;
    {
        // the slot's own pair, once: f_i0 -= fs e, f_i1 += fs e
        const float ex = q1.x - q0.x, ey = q1.y - q0.y, ez = q1.z - q0.z;
        const float r2 = ex * ex + ey * ey + ez * ez;
        if ((P == 1 || part == 0) && r2 < rc2) {
            float gx = 0.f, gy = 0.f, gz = 0.f, e = 0.f;
            unsigned k = 0;
            lj_term<ENERGY>(a.fc, ex, ey, ez, r2, gx, gy, gz, e, k);
            fx = make_float2(gx, -gx);
            fy = make_float2(gy, -gy);
            fz = make_float2(gz, -gz);
            if (ENERGY) {
                en = dup2(e);
                np0 = np1 = 1;
            }
        }
    }
    // the slot's atoms negated, in the two lanes of each pair
    const float2 nqx = make_float2(-q0.x, -q1.x), nqy = make_float2(-q0.y, -q1.y),
                 nqz = make_float2(-q0.z, -q1.z);
    const int nq = (min(p.count[s], p.cap) + 3) >> 2;
    const uint4 *lq = reinterpret_cast<const uint4 *>(p.list + list_group(s, p.cap)) + (s & 31);
    // one gather and one stencil shift per entry, both atoms' pair terms in
    // packed instructions; -fs = r2i s6 (e48 / 2 - e48 s6) is added with one fma
    auto pair = [&](uint32_t ent) {
        const float4 qj = __ldg(a.xq + (ent & kIndexMask));
        const float3 st = stencil_of(ent);
        const float tx = fmaf(st.x, w.x, qj.x), ty = fmaf(st.y, w.y, qj.y), tz = fmaf(st.z, w.z, qj.z);
        const float2 dx = add2(dup2(tx), nqx), dy = add2(dup2(ty), nqy), dz = add2(dup2(tz), nqz);
        const float2 r2 = fma2(dz, dz, fma2(dy, dy, mul2(dx, dx)));
        const float2 r2i = make_float2(rcp_fast(r2.x), rcp_fast(r2.y));
        const float2 s2 = mul2(dup2(a.fc.sig2f), r2i);
        const float2 s6 = mul2(mul2(s2, s2), s2);
        float2 nfs = mul2(mul2(fma2(s6, dup2(-a.fc.eps48f), dup2(0.5f * a.fc.eps48f)), s6), r2i);
        const bool in0 = r2.x < rc2, in1 = r2.y < rc2;
        nfs.x = in0 ? nfs.x : 0.f;
        nfs.y = in1 ? nfs.y : 0.f;
        fx = fma2(nfs, dx, fx);
        fy = fma2(nfs, dy, fy);
        fz = fma2(nfs, dz, fz);
        if (ENERGY) {
            float2 u = add2(mul2(fma2(s6, dup2(a.fc.eps4f), dup2(-a.fc.eps4f)), s6),
                            dup2(-a.fc.shiftf));
            u.x = in0 ? u.x : 0.f;
            u.y = in1 ? u.y : 0.f;
            en = add2(en, u);
            np0 += in0 ? 1u : 0u;
            np1 += in1 ? 1u : 0u;
        }
    };
    if constexpr (P > 1) {
        SplitState t, t1;
        load_slot_state<MODE, P>(a, i0, two, on, part, t, t1);
        split_quads<P>(lq, on ? nq : 0, part, pair);
        split_slot_out<MODE, ENERGY, false, P>(a, i0, two, on, part, fx, fy, fz, en, np0, np1, t, t1,
                                               store_f);
        return;
    }
    uint4 nxt = nq > 0 ? __ldcs(lq) : make_uint4(0u, 0u, 0u, 0u);
    for (int q = 0; q < nq; ++q) {
        const uint4 e4 = nxt;
        if (q + 1 < nq) nxt = __ldcs(lq + (size_t)(q + 1) * 32);
        pair(e4.x);
        pair(e4.y);
        pair(e4.z);
        pair(e4.w);
    }
    // the position words (id and species bits) are read again here rather
    // than held through the loop: registers are the kernel's limit
    pair_atom_out<MODE, ENERGY>(a, i0, fx.x, fy.x, fz.x, en.x, np0, a.xq[i0].w, store_f);
    if (two)
        pair_atom_out<MODE, ENERGY>(a, i0 + 1, fx.y, fy.y, fz.y, en.y, np1, a.xq[i0 + 1].w, store_f);
}

}  // namespace mdg
