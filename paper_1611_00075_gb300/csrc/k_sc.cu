// k_sc.cu -- Sutton-Chen many-body forces in the paper's three steps
// (Sec. 3.1): a pair pass for the localization function rho_i (Eq. 2), an
// atom pass for the embedding function, and a pair pass for the pair term
// and the forces.
//
// Sutton-Chen instance of Eq. 1:
//   Phi(r) = eps (a/r)^n,  psi(r) = (a/r)^m,  F(rho) = -eps c sqrt(rho),
//   truncated (no shift) at r_c.  Differentiating U gives the force on i
//   f_i = -sum_j [Phi'(r) + (F'(rho_i) + F'(rho_j)) psi'(r)] (r_i - r_j) / r
//       = -sum_j (n Phi + m (F'_i + F'_j) psi) / r^2 * d,   d = r_j - r_i
//   since Phi' = -n Phi / r and psi' = -m psi / r.
//
// The second step (atom loop: F(rho_i), F'(rho_i)) only needs rho_i, so it
// runs as the epilogue of the density pass in the thread that owns atom i;
// sc_embed_deriv_*() below is that step.  The third step needs F'_j per pair:
// the mixed path's density epilogue writes (x, y, z, F'(rho)) of each atom
// into one float4, so the force pass gathers position and F'_j in one load.
//
// Precision as for Lennard-Jones: MIXED computes pair terms in float32 and
// sums rho and the forces in float64 over float32 chunks; F'(rho) feeds the
// float32 pair terms as float32.  The embedding energy is float64.
#include "k_common.cuh"
#include "k_fp64.cuh"
#include "k_pair.cuh"

namespace mdg {

namespace {

template <int K>
__device__ __forceinline__ float cpow(float x) {
    float r = 1.f, b = x;
    int k = K;
#pragma unroll
    for (int t = 0; t < 6; ++t) {
        if (k & 1) r *= b;
        k >>= 1;
        if (k) b *= b;
    }
    return r;
}
__device__ __forceinline__ float rpow(float x, int k) {
    float r = 1.f;
    while (k) {
        if (k & 1) r *= x;
        k >>= 1;
        x *= x;
    }
    return r;
}
__device__ __forceinline__ double rpowd(double x, int k) {
    double r = 1.0;
    while (k) {
        if (k & 1) r *= x;
        k >>= 1;
        x *= x;
    }
    return r;
}

// Up to these sizes eight lanes share an atom or a slot.  One step (both passes),
// eight lanes against one, us: per-atom lists 16.5 / 39 at 1,372 atoms, 24.5 / 44
// at 6,912, 36 / 45 at 16,384, 56 / 46 at 32,000; slots of two 19.7 / 61, 23.7 /
// 82, 31 / 69, 48 / 72 and, at 55,296 atoms, 106 / 110.
constexpr int64_t kScSplitAtoms = 20480, kScSplitSlots = 24576;

// (a/r)^K from s = (a/r)^2 and ar = a/r (ar only used for odd K).
template <int K>
__device__ __forceinline__ float ar_pow(float s, float ar) {
    if (K % 2 == 0) return cpow<K / 2>(s);
    return cpow<K / 2>(s) * ar;
}

// The atom step of Sec. 3.1 for Sutton-Chen: F'(rho) = -eps c / (2 sqrt(rho)).
__device__ __forceinline__ float sc_embed_deriv_f32(double rho, float ec) {
    return rho > 0.0 ? -0.5f * ec * rsqrtf((float)rho) : 0.f;
}
__device__ __forceinline__ double sc_embed_deriv_f64(double rho, double ec) {
    return rho > 0.0 ? -0.5 * ec / sqrt(rho) : 0.0;
}

// Both mixed passes run 256-thread blocks at up to 64 registers (4 per SM),
// measured 2 % faster than at 48.
template <int ME, int P>
__global__ void __launch_bounds__(kBlock, P > 1 ? 1 : 4) sc_density_mixed(ForceArgs a) {
    if (a.ds->status != 0) return;
    const int tid = blockIdx.x * blockDim.x + threadIdx.x;
    const bool on = tid / P < a.n;
    if (P == 1 && !on) return;
    const int i = on ? tid / P : a.n - 1, part = tid % P;
    const float4 qi = a.xq[i];
    const int nq = (min(a.ncount[i], a.cap) + 3) >> 2;
    const uint4 *lq = reinterpret_cast<const uint4 *>(a.nlist + list_group(i, a.cap)) + (i & 31);
    const float rc2 = a.fc.rc2f, af = a.fc.sc_af, a2 = af * af;
    const int m = a.fc.sc_m;
    double R = 0.0;
    float r = 0.f;
    auto pair = [&](uint32_t ent) {
        const float4 qj = __ldg(a.xq + (ent & kIndexMask));
        const float3 st = stencil_of(ent);
        const float ex = fmaf(st.x, a.g.wf[0], qj.x - qi.x);
        const float ey = fmaf(st.y, a.g.wf[1], qj.y - qi.y);
        const float ez = fmaf(st.z, a.g.wf[2], qj.z - qi.z);
        const float r2 = dist2(ex, ey, ez);
        if (r2 < rc2) {
            const float s = a2 * rcp_fast(r2);
            float psi;
            if (ME > 0) psi = ar_pow<ME>(s, (ME & 1) ? af * rsqrt_fast(r2) : 0.f);
            else psi = (m & 1) ? rpow(s, m / 2) * af * rsqrt_fast(r2) : rpow(s, m / 2);
            r += psi;
        }
    };
    if (P > 1) {
        split_quads<P>(lq, on ? nq : 0, part, pair);
        R = split_sum<P>((double)r);
        if (!on || part != 0) return;
    } else {
        // list quads stream through once (evict-first), one quad loaded ahead
        uint4 nxt = nq > 0 ? __ldcs(lq) : make_uint4(0u, 0u, 0u, 0u);
        for (int q0 = 0; q0 < nq; q0 += kChunkQ) {
            const int q1 = min(q0 + kChunkQ, nq);
            r = 0.f;
            for (int q = q0; q < q1; ++q) {
                const uint4 e4 = nxt;
                if (q + 1 < nq) nxt = __ldcs(lq + (size_t)(q + 1) * 32);
                pair(e4.x);
                pair(e4.y);
                pair(e4.z);
                pair(e4.w);
            }
            R += (double)r;
        }
    }
    a.rho[i] = R;
    const float dF = sc_embed_deriv_f32(R, a.fc.sc_ecf);
    a.dF32[i] = dF;
    // the force pass gathers F'(rho_j) together with the position of j
    a.xqf[i] = make_float4(qi.x, qi.y, qi.z, dF);
}

// (a/r)^K in float64 from s = (a/r)^2, K = 0: the run-time exponent k; an odd
// exponent also takes ar = a/r.
template <int K>
__device__ __forceinline__ double ar_pow_f64(double s, double ar, int k) {
    if (K == 6) return s * s * s;
    if (K == 9) return (s * s) * (s * s) * ar;
    const double p = rpowd(s, k / 2);
    return (k & 1) ? p * ar : p;
}

// The float64 passes run the pair loop of k_fp64.cuh, P lanes per atom; NE, ME:
// the exponents 9 and 6 at compile time, or 0.
template <int NE, int ME, int P>
__global__ void __launch_bounds__(kF64Block) sc_density_fp64(ForceArgs a) {
    __shared__ ShiftTab sh;
    __shared__ Home64 home;
    load_shifts_f32(a.g, &sh);
    __syncthreads();
    if (a.ds->status != 0) return;
    const long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    const bool on = t < (long long)a.n * P;
    const int i = on ? (int)(t / P) : 0, part = (int)(t % P);
    double R = 0.0;
    load_home64<P>(a, i, part, &home);
    if (on) {
        const double A = a.fc.sc_a, A2 = A * A;
        const int m = a.fc.sc_m;
        const int seed_hi = a.fc.f64_seed_hi;
        f64_pairs<P>(a, &sh, &home, i, part, a.xq[i],
                     [&](int, double, double, double, double r2) {
                         if (ME > 0 ? (ME & 1) : (m & 1)) {
                             const double ar = A * rsqrt_f64(r2, seed_hi);
                             R += ar_pow_f64<ME>(ar * ar, ar, m);
                         } else {
                             R += ar_pow_f64<ME>(A2 * rcp_f64(r2, seed_hi), 0.0, m);
                         }
                     });
    }
    if (P > 1) R = lanes_sum<P>(R);
    if (!on || part != 0) return;
    a.rho[i] = R;
    const double d = sc_embed_deriv_f64(R, a.fc.sc_ec);
    a.dF64[i] = d;
    a.dF32[i] = (float)d;
}

template <int MODE, bool ENERGY, int NE, int ME, int P>
__global__ void __launch_bounds__(kBlock, P > 1 ? 1 : 4) sc_force_mixed(ForceArgs a, int store_f) {
    if (a.ds->status != 0) return;
    step_bookkeeping<MODE>(a);
    const int tid = blockIdx.x * blockDim.x + threadIdx.x;
    const bool on = tid / P < a.n;
    if (P == 1 && !on) return;
    const int i = on ? tid / P : a.n - 1, part = tid % P;
    const float4 qi = a.xqf[i];  // position, F'(rho_i)
    const float dFi = qi.w;
    const int nq = (min(a.ncount[i], a.cap) + 3) >> 2;
    const uint4 *lq = reinterpret_cast<const uint4 *>(a.nlist + list_group(i, a.cap)) + (i & 31);
    const float rc2 = a.fc.rc2f, af = a.fc.sc_af, a2 = af * af, epsf = a.fc.sc_epsf;
    const float inv_a2 = 1.0f / a2;
    const int nexp = a.fc.sc_n, mexp = a.fc.sc_m;
    const float nf = (float)(NE > 0 ? NE : nexp), mf = (float)(ME > 0 ? ME : mexp);
    double Fx = 0.0, Fy = 0.0, Fz = 0.0, E = 0.0;
    unsigned npair = 0;
    float fx = 0.f, fy = 0.f, fz = 0.f, e = 0.f;
    auto pair = [&](uint32_t ent) {
        const float4 qj = __ldg(a.xqf + (ent & kIndexMask));  // position, F'(rho_j)
        const float3 st = stencil_of(ent);
        const float ex = fmaf(st.x, a.g.wf[0], qj.x - qi.x);
        const float ey = fmaf(st.y, a.g.wf[1], qj.y - qi.y);
        const float ez = fmaf(st.z, a.g.wf[2], qj.z - qi.z);
        const float r2 = dist2(ex, ey, ez);
        if (r2 < rc2) {
            // with an odd exponent a/r comes from one reciprocal square
            // root, and (a/r)^2 and 1/r^2 from it without a reciprocal
            const bool odd = (NE > 0) ? ((NE | ME) & 1) : ((nexp | mexp) & 1);
            const float ar = odd ? af * rsqrt_fast(r2) : 0.f;
            const float r2i = odd ? ar * ar * inv_a2 : rcp_fast(r2);
            const float s = odd ? ar * ar : a2 * r2i;
            float Phi, psi;
            if (NE > 0) {
                Phi = epsf * ar_pow<NE>(s, ar);
                psi = ar_pow<ME>(s, ar);
            } else {
                Phi = epsf * ((nexp & 1) ? rpow(s, nexp / 2) * ar : rpow(s, nexp / 2));
                psi = (mexp & 1) ? rpow(s, mexp / 2) * ar : rpow(s, mexp / 2);
            }
            const float fs = (nf * Phi + mf * (dFi + qj.w) * psi) * r2i;
            fx -= fs * ex;
            fy -= fs * ey;
            fz -= fs * ez;
            if (ENERGY) {
                e += Phi;
                ++npair;
            }
        }
    };
    if constexpr (P > 1) {
        const int c = part & 3;
        const SplitState st = load_split_state<MODE>(a, i, c, on && part < 4);
        split_quads<P>(lq, on ? nq : 0, part, pair);
        Fx = split_sum<P>((double)fx);
        Fy = split_sum<P>((double)fy);
        Fz = split_sum<P>((double)fz);
        if (ENERGY) {
            E = split_sum<P>((double)e);
            if (on) count_pairs(a.ds, npair);
            if (on && part == 0) a.e_atom[i] = 0.5 * E - a.fc.sc_ec * sqrt(a.rho[i]);
        }
        split_epilogue<MODE>(a, i, c, on && part < 4, c == 0 ? Fx : (c == 1 ? Fy : Fz),
                             reinterpret_cast<const float *>(a.xq)[4 * (size_t)i + 3], st, store_f);
        return;
    }
    uint4 nxt = nq > 0 ? __ldcs(lq) : make_uint4(0u, 0u, 0u, 0u);
    for (int q0 = 0; q0 < nq; q0 += kChunkQ) {
        const int q1 = min(q0 + kChunkQ, nq);
        fx = fy = fz = e = 0.f;
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
        if (ENERGY) E += (double)e;
    }
    const size_t n = (size_t)a.n;
    if (MODE == FM_STORE || store_f) {
        a.f[i] = Fx;
        a.f[n + i] = Fy;
        a.f[2 * n + i] = Fz;
    }
    if (ENERGY) {
        a.e_atom[i] = 0.5 * E - a.fc.sc_ec * sqrt(a.rho[i]);
        count_pairs(a.ds, npair);
    }
    // the float32 position's w word holds the original id
    if (MODE != FM_STORE)
        vv_epilogue<MODE>(a, i, Fx, Fy, Fz, reinterpret_cast<const float *>(a.xq)[4 * (size_t)i + 3]);
}

template <int MODE, bool ENERGY, int NE, int ME, int P>
__global__ void __launch_bounds__(kF64Block) sc_force_fp64(ForceArgs a, int store_f) {
    __shared__ ShiftTab sh;
    __shared__ Home64 home;
    load_shifts_f32(a.g, &sh);
    __syncthreads();
    if (a.ds->status != 0) return;
    step_bookkeeping<MODE>(a);
    const long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    const bool on = t < (long long)a.n * P;
    const int i = on ? (int)(t / P) : 0, part = (int)(t % P);
    double fx = 0.0, fy = 0.0, fz = 0.0, e = 0.0;
    unsigned npair = 0;
    float qw = 0.f;
    load_home64<P>(a, i, part, &home);
    if (on) {
        const float4 qi = a.xq[i];
        qw = qi.w;
        const double dFi = a.dF64[i];
        const double A = a.fc.sc_a, A2 = A * A, eps = a.fc.sc_eps;
        const int nexp = a.fc.sc_n, mexp = a.fc.sc_m;
        const double nd = (double)(NE > 0 ? NE : nexp), mD = (double)(ME > 0 ? ME : mexp);
        const bool odd = NE > 0 ? ((NE | ME) & 1) : ((nexp | mexp) & 1);
        const int seed_hi = a.fc.f64_seed_hi;
        f64_pairs<P>(a, &sh, &home, i, part, qi,
                     [&](int j, double ex, double ey, double ez, double r2) {
                         double ar = 0.0, r2i;
                         if (odd) {
                             const double y = rsqrt_f64(r2, seed_hi);
                             ar = A * y;
                             r2i = y * y;
                         } else {
                             r2i = rcp_f64(r2, seed_hi);
                         }
                         const double s = A2 * r2i;
                         const double Phi = eps * ar_pow_f64<NE>(s, ar, nexp);
                         const double psi = ar_pow_f64<ME>(s, ar, mexp);
                         const double fs = (nd * Phi + mD * (dFi + a.dF64[j]) * psi) * r2i;
                         fx -= fs * ex;
                         fy -= fs * ey;
                         fz -= fs * ez;
                         if (ENERGY) {
                             e += Phi;
                             ++npair;
                         }
                     });
    }
    if (ENERGY) {
        e = lanes_sum<P>(e);
        if (on) count_pairs(a.ds, npair);
        if (on && part == 0) a.e_atom[i] = 0.5 * e - a.fc.sc_ec * sqrt(a.rho[i]);
    }
    f64_finish<MODE, false, P>(a, i, part, on, fx, fy, fz, qw, store_f);
}

template <int NE, int ME, int P>
cudaError_t launch_sc_fp64(const ForceArgs &a, bool density, int mode, bool energy, int sf,
                           cudaStream_t s) {
    const int nb = nblocks((int64_t)a.n * P, kF64Block);
    if (density) {
        sc_density_fp64<NE, ME, P><<<nb, kF64Block, 0, s>>>(a);
        return cudaGetLastError();
    }
    switch (mode) {
        case FM_STORE:
            if (energy) sc_force_fp64<FM_STORE, true, NE, ME, P><<<nb, kF64Block, 0, s>>>(a, sf);
            else sc_force_fp64<FM_STORE, false, NE, ME, P><<<nb, kF64Block, 0, s>>>(a, sf);
            break;
        case FM_FUSED_FULL:
            sc_force_fp64<FM_FUSED_FULL, false, NE, ME, P><<<nb, kF64Block, 0, s>>>(a, sf);
            break;
        default: sc_force_fp64<FM_FUSED_HALF, false, NE, ME, P><<<nb, kF64Block, 0, s>>>(a, sf); break;
    }
    return cudaGetLastError();
}

// the pass (density or force) in float64, its lanes per atom by size
cudaError_t launch_sc_fp64_any(const ForceArgs &a, bool density, int mode, bool energy, int sf,
                               cudaStream_t s) {
    const bool cu = a.fc.sc_n == 9 && a.fc.sc_m == 6;
#define MDG_SC64(P)                                                                   \
    (cu ? launch_sc_fp64<9, 6, P>(a, density, mode, energy, sf, s)                    \
        : launch_sc_fp64<0, 0, P>(a, density, mode, energy, sf, s))
    switch (f64_split(a.n)) {
        case 1: return MDG_SC64(1);
        case 4: return MDG_SC64(4);
        case 8: return MDG_SC64(8);
        default: return MDG_SC64(16);
    }
#undef MDG_SC64
}

// ---- two atoms per thread (MD_FORCE_PAIRED) ---------------------------------
//
// The slot layout of k_pair.cu: slot s holds sorted atoms i0 and i0 + 1 of
// one cell (one atom when bit 31 of its entry is set) and the union of their
// lists.  Both passes evaluate the slot's own pair once, then both atoms
// against each list entry with packed float32 pairs (lane x: i0, lane y:
// i1), so that one gathered neighbour serves two pair evaluations.  Sums run
// in float32 over chunks of kChunkQ quads and in float64 across chunks, as in
// the per-atom passes: a crystal's many-body forces cancel strongly.
constexpr int kScPairBlock = 128;

// (a/r)^K lane by lane for run-time exponents (s = (a/r)^2, ar = a/r)
__device__ __forceinline__ float2 ar_pow_rt(float2 s, float2 ar, int k) {
    float2 r = make_float2(rpow(s.x, k / 2), rpow(s.y, k / 2));
    if (k & 1) r = mul2(r, ar);
    return r;
}

template <int ME, int P>
__global__ void __launch_bounds__(kScPairBlock, P > 1 ? 1 : 8) sc_density_pair(ForceArgs a, PairArgs p) {
    if (a.ds->status != 0) return;
    const int tid = blockIdx.x * blockDim.x + threadIdx.x;
    const int nslots = p.slot_start[p.ncells];
    if ((P > 1 ? (tid & ~31) / P : tid) >= nslots) return;  // P > 1: whole warps
    const bool on = tid / P < nslots;
    const int s = on ? tid / P : nslots - 1, part = tid % P;
    const uint32_t sa = p.slot_atom[s];
    const int i0 = (int)(sa & ~kSingle);
    const bool two = !(sa & kSingle);
    const float4 q0 = a.xq[i0];
    const float4 q1 = two ? a.xq[i0 + 1] : make_float4(3.0e18f, 3.0e18f, 3.0e18f, 0.f);
    const float rc2 = a.fc.rc2f, af = a.fc.sc_af, a2 = af * af;
    const int m = a.fc.sc_m;
    float2 r = dup2(0.f);
    {
        // the slot's own pair adds to both densities
        const float ex = q1.x - q0.x, ey = q1.y - q0.y, ez = q1.z - q0.z;
        const float r2 = ex * ex + ey * ey + ez * ez;
        if (part == 0 && r2 < rc2) {
            const float sp = a2 * rcp_fast(r2);
            const float psi = ME > 0 ? ar_pow<ME>(sp, (ME & 1) ? af * rsqrt_fast(r2) : 0.f)
                                     : ((m & 1) ? rpow(sp, m / 2) * af * rsqrt_fast(r2)
                                                : rpow(sp, m / 2));
            r = dup2(psi);
        }
    }
    const float2 nqx = make_float2(-q0.x, -q1.x), nqy = make_float2(-q0.y, -q1.y),
                 nqz = make_float2(-q0.z, -q1.z);
    const int nq = (min(p.count[s], p.cap) + 3) >> 2;
    const uint4 *lq = reinterpret_cast<const uint4 *>(p.list + list_group(s, p.cap)) + (s & 31);
    auto pair = [&](uint32_t ent) {
        const float4 qj = __ldg(a.xq + (ent & kIndexMask));
        const float3 st = stencil_of(ent);
        const float tx = fmaf(st.x, a.g.wf[0], qj.x), ty = fmaf(st.y, a.g.wf[1], qj.y), tz = fmaf(st.z, a.g.wf[2], qj.z);
        const float2 dx = add2(dup2(tx), nqx), dy = add2(dup2(ty), nqy), dz = add2(dup2(tz), nqz);
        const float2 r2 = fma2(dz, dz, fma2(dy, dy, mul2(dx, dx)));
        const float2 sp = mul2(dup2(a2), make_float2(rcp_fast(r2.x), rcp_fast(r2.y)));
        float2 psi;
        if (ME == 6) {
            psi = mul2(mul2(sp, sp), sp);
        } else {
            const float2 ar = (m & 1) ? make_float2(af * rsqrt_fast(r2.x), af * rsqrt_fast(r2.y)) : dup2(0.f);
            psi = ar_pow_rt(sp, ar, m);
        }
        psi.x = r2.x < rc2 ? psi.x : 0.f;
        psi.y = r2.y < rc2 ? psi.y : 0.f;
        r = add2(r, psi);
    };
    double R0 = 0.0, R1 = 0.0;
    if (P > 1) {
        split_quads<P>(lq, on ? nq : 0, part, pair);
        R0 = split_sum<P>((double)r.x);
        R1 = split_sum<P>((double)r.y);
        if (!on || part != 0) return;
        r = dup2(0.f);
    }
    uint4 nxt = nq > 0 ? __ldcs(lq) : make_uint4(0u, 0u, 0u, 0u);
    for (int c0 = 0; P == 1 && c0 < nq; c0 += kChunkQ) {
        const int c1 = min(c0 + kChunkQ, nq);
        for (int q = c0; q < c1; ++q) {
            const uint4 e4 = nxt;
            if (q + 1 < nq) nxt = __ldcs(lq + (size_t)(q + 1) * 32);
            pair(e4.x);
            pair(e4.y);
            pair(e4.z);
            pair(e4.w);
        }
        R0 += (double)r.x;
        R1 += (double)r.y;
        r = dup2(0.f);
    }
    R0 += (double)r.x;
    R1 += (double)r.y;
    // the atom step (embedding derivative) and the gather record of the force pass
    const float d0 = sc_embed_deriv_f32(R0, a.fc.sc_ecf);
    a.rho[i0] = R0;
    a.dF32[i0] = d0;
    a.xqf[i0] = make_float4(q0.x, q0.y, q0.z, d0);
    if (two) {
        const float d1 = sc_embed_deriv_f32(R1, a.fc.sc_ecf);
        a.rho[i0 + 1] = R1;
        a.dF32[i0 + 1] = d1;
        a.xqf[i0 + 1] = make_float4(q1.x, q1.y, q1.z, d1);
    }
}

template <int MODE, bool ENERGY>
__device__ __forceinline__ void sc_pair_atom_out(const ForceArgs &a, int i, double Fx, double Fy,
                                                 double Fz, double E, unsigned np, int store_f) {
    const size_t n = (size_t)a.n;
    if (MODE == FM_STORE || store_f) {
        a.f[i] = Fx;
        a.f[n + i] = Fy;
        a.f[2 * n + i] = Fz;
    }
    if (ENERGY) {
        a.e_atom[i] = 0.5 * E - a.fc.sc_ec * sqrt(a.rho[i]);
        count_pairs(a.ds, np);
    }
    // the float32 position's w word holds the original id
    if (MODE != FM_STORE)
        vv_epilogue<MODE>(a, i, Fx, Fy, Fz, reinterpret_cast<const float *>(a.xq)[4 * (size_t)i + 3]);
}

template <int MODE, bool ENERGY, int NE, int ME, int P>
__global__ void __launch_bounds__(kScPairBlock, P > 1 ? 1 : 7) sc_force_pair(ForceArgs a, PairArgs p,
                                                                 int store_f) {
    if (a.ds->status != 0) return;
    step_bookkeeping<MODE>(a);
    const int tid = blockIdx.x * blockDim.x + threadIdx.x;
    const int nslots = p.slot_start[p.ncells];
    if ((P > 1 ? (tid & ~31) / P : tid) >= nslots) return;  // P > 1: whole warps
    const bool on = tid / P < nslots;
    const int s = on ? tid / P : nslots - 1, part = tid % P;
    const uint32_t sa = p.slot_atom[s];
    const int i0 = (int)(sa & ~kSingle);
    const bool two = !(sa & kSingle);
    const float4 q0 = a.xqf[i0];  // position, F'(rho)
    const float4 q1 = two ? a.xqf[i0 + 1] : make_float4(3.0e18f, 3.0e18f, 3.0e18f, 0.f);
    const float2 dFi = make_float2(q0.w, q1.w);
    const float rc2 = a.fc.rc2f, af = a.fc.sc_af, a2 = af * af, epsf = a.fc.sc_epsf;
    const float inv_a2 = 1.0f / a2;
    const int nexp = a.fc.sc_n, mexp = a.fc.sc_m;
    const float nf = (float)(NE > 0 ? NE : nexp), mf = (float)(ME > 0 ? ME : mexp);
    const bool odd = (NE > 0) ? ((NE | ME) & 1) : ((nexp | mexp) & 1);
    float2 fx = dup2(0.f), fy = dup2(0.f), fz = dup2(0.f), en = dup2(0.f);
    unsigned np0 = 0, np1 = 0;
    {
        // the slot's own pair once: e = x_1 - x_0, f_0 -= fs e, f_1 += fs e
        const float ex = q1.x - q0.x, ey = q1.y - q0.y, ez = q1.z - q0.z;
        const float r2 = ex * ex + ey * ey + ez * ez;
        if (part == 0 && r2 < rc2) {
            const float r2i = rcp_fast(r2);
            const float sp = a2 * r2i;
            const float ar = odd ? af * rsqrt_fast(r2) : 0.f;
            float Phi, psi;
            if (NE > 0) {
                Phi = epsf * ar_pow<NE>(sp, ar);
                psi = ar_pow<ME>(sp, ar);
            } else {
                Phi = epsf * ((nexp & 1) ? rpow(sp, nexp / 2) * ar : rpow(sp, nexp / 2));
                psi = (mexp & 1) ? rpow(sp, mexp / 2) * ar : rpow(sp, mexp / 2);
            }
            const float fs = (nf * Phi + mf * (q0.w + q1.w) * psi) * r2i;
            fx = make_float2(-fs * ex, fs * ex);
            fy = make_float2(-fs * ey, fs * ey);
            fz = make_float2(-fs * ez, fs * ez);
            if (ENERGY) {
                en = dup2(Phi);
                np0 = np1 = 1;
            }
        }
    }
    const float2 nqx = make_float2(-q0.x, -q1.x), nqy = make_float2(-q0.y, -q1.y),
                 nqz = make_float2(-q0.z, -q1.z);
    const int nq = (min(p.count[s], p.cap) + 3) >> 2;
    const uint4 *lq = reinterpret_cast<const uint4 *>(p.list + list_group(s, p.cap)) + (s & 31);
    // d = x_j - x_i per atom; f_i -= fs d with fs = (n Phi + m (F'_i + F'_j) psi) / r^2
    auto pair = [&](uint32_t ent) {
        const float4 qj = __ldg(a.xqf + (ent & kIndexMask));  // position, F'(rho_j)
        const float3 st = stencil_of(ent);
        const float tx = fmaf(st.x, a.g.wf[0], qj.x), ty = fmaf(st.y, a.g.wf[1], qj.y), tz = fmaf(st.z, a.g.wf[2], qj.z);
        const float2 dx = add2(dup2(tx), nqx), dy = add2(dup2(ty), nqy), dz = add2(dup2(tz), nqz);
        const float2 r2 = fma2(dz, dz, fma2(dy, dy, mul2(dx, dx)));
        // with an odd exponent a/r comes from one reciprocal square root,
        // and (a/r)^2 and 1/r^2 from it without a reciprocal
        float2 ar, sp, r2i;
        if (odd) {
            ar = mul2(dup2(af), make_float2(rsqrt_fast(r2.x), rsqrt_fast(r2.y)));
            sp = mul2(ar, ar);
            r2i = mul2(sp, dup2(inv_a2));
        } else {
            ar = dup2(0.f);
            r2i = make_float2(rcp_fast(r2.x), rcp_fast(r2.y));
            sp = mul2(dup2(a2), r2i);
        }
        float2 Phi, psi;
        if (NE == 9 && ME == 6) {
            const float2 s2 = mul2(sp, sp);
            psi = mul2(s2, sp);
            Phi = mul2(mul2(mul2(s2, s2), ar), dup2(epsf));
        } else {
            Phi = mul2(dup2(epsf), ar_pow_rt(sp, ar, NE > 0 ? NE : nexp));
            psi = ar_pow_rt(sp, ar, ME > 0 ? ME : mexp);
        }
        const float2 t = add2(dFi, dup2(qj.w));
        float2 nfs = mul2(fma2(mul2(dup2(-mf), t), psi, mul2(dup2(-nf), Phi)), r2i);
        const bool in0 = r2.x < rc2, in1 = r2.y < rc2;
        nfs.x = in0 ? nfs.x : 0.f;
        nfs.y = in1 ? nfs.y : 0.f;
        fx = fma2(nfs, dx, fx);
        fy = fma2(nfs, dy, fy);
        fz = fma2(nfs, dz, fz);
        if (ENERGY) {
            en.x += in0 ? Phi.x : 0.f;
            en.y += in1 ? Phi.y : 0.f;
            np0 += in0 ? 1u : 0u;
            np1 += in1 ? 1u : 0u;
        }
    };
    if constexpr (P > 1) {
        SplitState st, st1;
        load_slot_state<MODE, P>(a, i0, two, on, part, st, st1);
        split_quads<P>(lq, on ? nq : 0, part, pair);
        const double F0[3] = {split_sum<P>((double)fx.x), split_sum<P>((double)fy.x),
                              split_sum<P>((double)fz.x)};
        const double F1[3] = {split_sum<P>((double)fx.y), split_sum<P>((double)fy.y),
                              split_sum<P>((double)fz.y)};
        if (ENERGY) {
            const double E0 = split_sum<P>((double)en.x), E1 = split_sum<P>((double)en.y);
            if (on) count_pairs(a.ds, np0 + (two ? np1 : 0u));
            if (on && part == 0) a.e_atom[i0] = 0.5 * E0 - a.fc.sc_ec * sqrt(a.rho[i0]);
            if (on && two && part == 1) a.e_atom[i0 + 1] = 0.5 * E1 - a.fc.sc_ec * sqrt(a.rho[i0 + 1]);
        }
        split_slot_finish<MODE, false, P>(a, i0, two, on, part, F0, F1, st, st1, store_f);
        return;
    }
    double F0x = 0.0, F0y = 0.0, F0z = 0.0, F1x = 0.0, F1y = 0.0, F1z = 0.0, E0 = 0.0, E1 = 0.0;
    auto flush = [&]() {
        F0x += (double)fx.x; F0y += (double)fy.x; F0z += (double)fz.x;
        F1x += (double)fx.y; F1y += (double)fy.y; F1z += (double)fz.y;
        fx = fy = fz = dup2(0.f);
        if (ENERGY) {
            E0 += (double)en.x;
            E1 += (double)en.y;
            en = dup2(0.f);
        }
    };
    uint4 nxt = nq > 0 ? __ldcs(lq) : make_uint4(0u, 0u, 0u, 0u);
    for (int c0 = 0; c0 < nq; c0 += kChunkQ) {
        const int c1 = min(c0 + kChunkQ, nq);
        for (int q = c0; q < c1; ++q) {
            const uint4 e4 = nxt;
            if (q + 1 < nq) nxt = __ldcs(lq + (size_t)(q + 1) * 32);
            pair(e4.x);
            pair(e4.y);
            pair(e4.z);
            pair(e4.w);
        }
        flush();
    }
    flush();
    sc_pair_atom_out<MODE, ENERGY>(a, i0, F0x, F0y, F0z, E0, np0, store_f);
    if (two) sc_pair_atom_out<MODE, ENERGY>(a, i0 + 1, F1x, F1y, F1z, E1, np1, store_f);
}

}  // namespace

cudaError_t launch_sc_density(md_system *h) {
    ForceArgs a = make_force_args(h);
    if (h->p.force_variant == MD_FORCE_PAIRED) {
        const PairArgs p = make_pair_args(h);
        const int P = split8(h->n / 2, h->ps_cap, kScSplitSlots);
        const bool six = a.fc.sc_m == 6;
        auto k = P > 1 ? (six ? sc_density_pair<6, 8> : sc_density_pair<0, 8>)
                       : (six ? sc_density_pair<6, 1> : sc_density_pair<0, 1>);
        k<<<pair_grid_blocks(h, kScPairBlock, P), kScPairBlock, 0, h->stream>>>(a, p);
        return cudaGetLastError();
    }
    if (h->p.precision == MD_MIXED) {
        const int P = split8(h->n, h->cap, kScSplitAtoms);
        const bool six = a.fc.sc_m == 6;
        auto k = P > 1 ? (six ? sc_density_mixed<6, 8> : sc_density_mixed<0, 8>)
                       : (six ? sc_density_mixed<6, 1> : sc_density_mixed<0, 1>);
        k<<<nblocks(h->n * P), kBlock, 0, h->stream>>>(a);
    } else {
        return launch_sc_fp64_any(a, true, FM_STORE, false, 0, h->stream);
    }
    return cudaGetLastError();
}

cudaError_t launch_sc_force(md_system *h, int mode, bool energy, bool store_f) {
    ForceArgs a = make_force_args(h);
    const int sf = store_f ? 1 : 0;
    cudaStream_t s = h->stream;
    if (h->p.force_variant == MD_FORCE_PAIRED) {
        const PairArgs p = make_pair_args(h);
        const int P = split8(h->n / 2, h->ps_cap, kScSplitSlots);
        const int pb = pair_grid_blocks(h, kScPairBlock, P);
        const bool cu = (a.fc.sc_n == 9 && a.fc.sc_m == 6);
#define MDG_SCP(M, E)                                                                   \
    do {                                                                                \
        auto k = P > 1 ? (cu ? sc_force_pair<M, E, 9, 6, 8> : sc_force_pair<M, E, 0, 0, 8>)  \
                       : (cu ? sc_force_pair<M, E, 9, 6, 1> : sc_force_pair<M, E, 0, 0, 1>); \
        k<<<pb, kScPairBlock, 0, s>>>(a, p, sf);                                        \
    } while (0)
        switch (mode) {
            case FM_STORE: if (energy) MDG_SCP(FM_STORE, true); else MDG_SCP(FM_STORE, false); break;
            case FM_FUSED_FULL: if (energy) MDG_SCP(FM_FUSED_FULL, true); else MDG_SCP(FM_FUSED_FULL, false); break;
            default: if (energy) MDG_SCP(FM_FUSED_HALF, true); else MDG_SCP(FM_FUSED_HALF, false); break;
        }
#undef MDG_SCP
        return cudaGetLastError();
    }
    if (h->p.precision == MD_MIXED) {
        const int P = split8(h->n, h->cap, kScSplitAtoms);
        const bool cu = (a.fc.sc_n == 9 && a.fc.sc_m == 6);
#define MDG_SC(M, E)                                                                    \
    do {                                                                                \
        auto k = P > 1 ? (cu ? sc_force_mixed<M, E, 9, 6, 8> : sc_force_mixed<M, E, 0, 0, 8>)  \
                       : (cu ? sc_force_mixed<M, E, 9, 6, 1> : sc_force_mixed<M, E, 0, 0, 1>); \
        k<<<nblocks(h->n * P), kBlock, 0, s>>>(a, sf);                                  \
    } while (0)
        switch (mode) {
            case FM_STORE: if (energy) MDG_SC(FM_STORE, true); else MDG_SC(FM_STORE, false); break;
            case FM_FUSED_FULL: if (energy) MDG_SC(FM_FUSED_FULL, true); else MDG_SC(FM_FUSED_FULL, false); break;
            default: if (energy) MDG_SC(FM_FUSED_HALF, true); else MDG_SC(FM_FUSED_HALF, false); break;
        }
#undef MDG_SC
    } else {
        return launch_sc_fp64_any(a, false, mode, energy, sf, s);
    }
    return cudaGetLastError();
}

}  // namespace mdg
