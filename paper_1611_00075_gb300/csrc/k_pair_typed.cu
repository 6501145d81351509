// k_pair_typed.cu -- two home atoms per thread (MD_FORCE_PAIRED) for the
// multi-element Lennard-Jones systems (Sec. 2.2's parameter reload, the
// Alloy and Layer configurations of Sec. 3.1).
//
// The slots and union lists of k_pair.cu, unchanged: a slot's two atoms may
// be of different species.  Each thread keeps the parameter rows of both of
// its atoms' species in registers (sigma^2 and 48 eps, with the energy 4 eps
// and the shift at r_c for energies); per list entry it reads the
// neighbour's species from the position word it gathers anyway and picks
// the two atoms' parameters from their rows, so each lane of the packed
// float32 pair arithmetic carries its own pair's parameters.  Sums: float32
// over the whole list, as for the one-species slot kernel; the
// velocity-Verlet epilogue uses each atom's species mass.
#include <cstring>

#include "k_pair.cuh"

namespace mdg {

namespace {

constexpr int kTypedPairBlock = 128;

// 1 below the cutoff (r2 < rc2), else 0, on the multiply-add pipe: the saturated
// (rc2 - r2) 2^k, with 2^k = big at least 1 / ulp(rc2), in one multiply-add whose
// rounding keeps the sign (rb = rc2 2^k; both exact).  NaN gives 0.  A compare
// and a select per lane run on the half-rate ALU pipe, which the species selects
// already load: 1.15 M alloy atoms, 50 steps, 11.10 -> 10.60 ms.  (The one-species
// and Sutton-Chen slot kernels have no ALU selects to relieve and lose by the
// two registers: liquid 7.03 -> 7.14 ms, Sutton-Chen 33.2 -> 33.5.)
__device__ __forceinline__ float inside(float r2, float big, float rb) {
    float w;
    asm("fma.rn.sat.f32 %0, %1, %2, %3;" : "=f"(w) : "f"(r2), "f"(-big), "f"(rb));
    return w;
}
// biased exponent of rc2 for which 2^k of inside() is a normal number with room
__host__ __device__ __forceinline__ bool inside_fits(unsigned exponent) {
    return exponent >= 40 && exponent <= 200;
}
__device__ __forceinline__ float inside_scale(float rc2) {
    return __uint_as_float((284u - (__float_as_uint(rc2) >> 23)) << 23);
}

// element t of a row of NT values held in registers
template <int NT>
__device__ __forceinline__ float row_at(const float *row, int t) {
    if (NT == 1) return row[0];
    if (NT == 2) return t ? row[1] : row[0];
    if (NT == 3) return t == 0 ? row[0] : (t == 1 ? row[1] : row[2]);
    return t < 2 ? (t == 0 ? row[0] : row[1]) : (t == 2 ? row[2] : row[3]);
}

// row ti of an NT x NT parameter table into registers
template <int NT>
__device__ __forceinline__ void row_of(const float *tab, int ti, float *row) {
#pragma unroll
    for (int k = 0; k < NT; ++k) {
        float v = tab[k];
#pragma unroll
        for (int r = 1; r < NT; ++r) v = (ti == r) ? tab[r * NT + k] : v;
        row[k] = v;
    }
}

template <int MODE, bool ENERGY>
__device__ __forceinline__ void typed_atom_out(const ForceArgs &a, int i, double Fx, double Fy,
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
    if (MODE != FM_STORE) vv_epilogue<MODE, true>(a, i, Fx, Fy, Fz, qw);
}

// Seven CTAs per SM: 10.06 ms (alloy of 1.15 M atoms, whole run) against 10.66 at
// eight and 10.88 at six.
// P > 1: thread t serves slot t / P (as lj_pair_kernel).  SAT: the cutoff by
// inside(); false in units whose rc2 leaves it no room.
template <int MODE, bool ENERGY, int NT, int P, bool SAT>
__global__ void __launch_bounds__(kTypedPairBlock, P > 1 ? 1 : 7)
lj_typed_pair_kernel(ForceArgs a, PairArgs p, TypeTab tt, int store_f) {
    if (a.ds->status != 0) return;
    step_bookkeeping<MODE>(a);
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    const int nslots = p.slot_start[p.ncells];
    if ((P > 1 ? (t & ~31) / P : t) >= nslots) return;  // P > 1: whole warps
    const bool on = t / P < nslots;
    const int s = on ? t / P : nslots - 1, part = t % P;
    const uint32_t sa = p.slot_atom[s];
    const int i0 = (int)(sa & ~kSingle);
    const bool two = !(sa & kSingle);
    const float4 q0 = a.xq[i0];
    // a one-atom slot puts its second atom at the dummy's distance
    const float4 q1 = two ? a.xq[i0 + 1] : make_float4(3.0e18f, 3.0e18f, 3.0e18f, 0.f);
    const int t0 = species_of(__float_as_uint(q0.w));
    const int t1 = two ? species_of(__float_as_uint(q1.w)) : t0;
    float s2a[NT], s2b[NT], e48a[NT], e48b[NT];
    row_of<NT>(tt.s2, t0, s2a);
    row_of<NT>(tt.s2, t1, s2b);
    row_of<NT>(tt.e48, t0, e48a);
    row_of<NT>(tt.e48, t1, e48b);
    float e4a[ENERGY ? NT : 1], e4b[ENERGY ? NT : 1], sha[ENERGY ? NT : 1], shb[ENERGY ? NT : 1];
    if (ENERGY) {
        row_of<NT>(tt.e4, t0, e4a);
        row_of<NT>(tt.e4, t1, e4b);
        row_of<NT>(tt.sh, t0, sha);
        row_of<NT>(tt.sh, t1, shb);
    }
    const float rc2 = a.fc.rc2f;
    const float big = SAT ? inside_scale(rc2) : 0.f, rb = rc2 * big;
    float2 fx = dup2(0.f), fy = dup2(0.f), fz = dup2(0.f), en = dup2(0.f);
    unsigned np0 = 0, np1 = 0;
    {
        // the slot's own pair once: f_0 -= fs e, f_1 += fs e with e = x_1 - x_0
        const float ex = q1.x - q0.x, ey = q1.y - q0.y, ez = q1.z - q0.z;
        const float r2 = ex * ex + ey * ey + ez * ez;
        if (part == 0 && r2 < rc2) {
            const float r2i = rcp_fast(r2);
            float s6 = row_at<NT>(s2a, t1) * r2i;
            s6 = s6 * s6 * s6;
            const float fs = row_at<NT>(e48a, t1) * r2i * s6 * (s6 - 0.5f);
            fx = make_float2(-fs * ex, fs * ex);
            fy = make_float2(-fs * ey, fs * ey);
            fz = make_float2(-fs * ez, fs * ez);
            if (ENERGY) {
                en = dup2(row_at<NT>(e4a, t1) * s6 * (s6 - 1.0f) - row_at<NT>(sha, t1));
                np0 = np1 = 1;
            }
        }
    }
    const float2 nqx = make_float2(-q0.x, -q1.x), nqy = make_float2(-q0.y, -q1.y),
                 nqz = make_float2(-q0.z, -q1.z);
    const int nq = (min(p.count[s], p.cap) + 3) >> 2;
    const uint4 *lq = reinterpret_cast<const uint4 *>(p.list + list_group(s, p.cap)) + (s & 31);
    // -fs = 48 eps r2i s6 (1/2 - s6), s6 = (sigma^2 r2i)^3, each lane with its
    // own pair's sigma and eps
    auto pair = [&](uint32_t ent) {
        const float4 qj = __ldg(a.xq + (ent & kIndexMask));
        const float3 st = stencil_of(ent);
        const int tj = species_of(__float_as_uint(qj.w));
        const float tx = fmaf(st.x, a.g.wf[0], qj.x), ty = fmaf(st.y, a.g.wf[1], qj.y), tz = fmaf(st.z, a.g.wf[2], qj.z);
        const float2 dx = add2(dup2(tx), nqx), dy = add2(dup2(ty), nqy), dz = add2(dup2(tz), nqz);
        const float2 r2 = fma2(dz, dz, fma2(dy, dy, mul2(dx, dx)));
        const float2 r2i = make_float2(rcp_fast(r2.x), rcp_fast(r2.y));
        const float2 s2 = mul2(make_float2(row_at<NT>(s2a, tj), row_at<NT>(s2b, tj)), r2i);
        const float2 s6 = mul2(mul2(s2, s2), s2);
        const float2 e48 = make_float2(row_at<NT>(e48a, tj), row_at<NT>(e48b, tj));
        float2 nfs = mul2(mul2(mul2(e48, fma2(s6, dup2(-1.0f), dup2(0.5f))), s6), r2i);
        float2 in;
        if (SAT) {
            in = make_float2(inside(r2.x, big, rb), inside(r2.y, big, rb));
            nfs = mul2(nfs, in);
        } else {
            in = make_float2(r2.x < rc2 ? 1.f : 0.f, r2.y < rc2 ? 1.f : 0.f);
            nfs.x = r2.x < rc2 ? nfs.x : 0.f;
            nfs.y = r2.y < rc2 ? nfs.y : 0.f;
        }
        fx = fma2(nfs, dx, fx);
        fy = fma2(nfs, dy, fy);
        fz = fma2(nfs, dz, fz);
        if (ENERGY) {
            float2 u = add2(mul2(mul2(make_float2(row_at<NT>(e4a, tj), row_at<NT>(e4b, tj)),
                                      add2(s6, dup2(-1.0f))), s6),
                            make_float2(-row_at<NT>(sha, tj), -row_at<NT>(shb, tj)));
            en = fma2(u, in, en);
            np0 += in.x > 0.f ? 1u : 0u;
            np1 += in.y > 0.f ? 1u : 0u;
        }
    };
    if constexpr (P > 1) {
        SplitState st, st1;
        load_slot_state<MODE, P>(a, i0, two, on, part, st, st1);
        split_quads<P>(lq, on ? nq : 0, part, pair);
        split_slot_out<MODE, ENERGY, true, P>(a, i0, two, on, part, fx, fy, fz, en, np0, np1, st, st1,
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
    // than held through the loop
    typed_atom_out<MODE, ENERGY>(a, i0, fx.x, fy.x, fz.x, en.x, np0, a.xq[i0].w, store_f);
    if (two)
        typed_atom_out<MODE, ENERGY>(a, i0 + 1, fx.y, fy.y, fz.y, en.y, np1, a.xq[i0 + 1].w,
                                     store_f);
}

template <int NT, int P, bool SAT = true>
cudaError_t launch_nt(md_system *h, int mode, bool energy, bool store_f) {
    const ForceArgs a = make_force_args(h);
    const PairArgs p = make_pair_args(h);
    const TypeTab &tt = h->types;
    const int blocks = pair_grid_blocks(h, kTypedPairBlock, P);
    const int sf = store_f ? 1 : 0;
    cudaStream_t s = h->stream;
    switch (mode) {
        case FM_STORE:
            if (energy)
                lj_typed_pair_kernel<FM_STORE, true, NT, P, SAT><<<blocks, kTypedPairBlock, 0, s>>>(a, p, tt, sf);
            else
                lj_typed_pair_kernel<FM_STORE, false, NT, P, SAT><<<blocks, kTypedPairBlock, 0, s>>>(a, p, tt, sf);
            break;
        case FM_FUSED_FULL:
            lj_typed_pair_kernel<FM_FUSED_FULL, false, NT, P, SAT><<<blocks, kTypedPairBlock, 0, s>>>(a, p, tt, sf);
            break;
        default:
            lj_typed_pair_kernel<FM_FUSED_HALF, false, NT, P, SAT><<<blocks, kTypedPairBlock, 0, s>>>(a, p, tt, sf);
            break;
    }
    return cudaGetLastError();
}

template <int NT>
cudaError_t launch_any(md_system *h, int mode, bool energy, bool store_f) {
    unsigned bits;
    std::memcpy(&bits, &h->fc.rc2f, sizeof bits);
    if (!inside_fits(bits >> 23)) return launch_nt<NT, 1, false>(h, mode, energy, store_f);
    return split8(h->n / 2, h->ps_cap, kTypedSplit) > 1 ? launch_nt<NT, 8>(h, mode, energy, store_f)
                                                : launch_nt<NT, 1>(h, mode, energy, store_f);
}

}  // namespace

cudaError_t launch_pair_typed_forces(md_system *h, int mode, bool energy, bool store_f) {
    switch (h->fc.ntypes) {
        case 1: return launch_any<1>(h, mode, energy, store_f);
        case 2: return launch_any<2>(h, mode, energy, store_f);
        case 3: return launch_any<3>(h, mode, energy, store_f);
        default: return launch_any<4>(h, mode, energy, store_f);
    }
}

}  // namespace mdg
