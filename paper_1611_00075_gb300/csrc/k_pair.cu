// k_pair.cu -- two home atoms per thread (MD_FORCE_PAIRED).
//
// Sec. 4.1 contrasts the paper's per-atom SIMD pair loop with clustering:
// grouping atoms lets one neighbour load serve several pair evaluations,
// which avoids the gather cost that dominates light potentials.  Full 8 x 4
// cluster pairs waste most of their slots at r_c = 2.5 sigma (their bounding
// boxes are as large as the cut-off sphere); this layout clusters only the
// home side, and only by two: the atoms of each cell, in their sorted order,
// are taken two at a time into slots (a cell of odd occupancy ends with a
// one-atom slot).  A slot's list is the union of its two atoms' lists, so one
// gather of a neighbour position feeds two pair evaluations: the union of two
// r_list spheres about one atom spacing apart holds about 1.3 times the
// entries of one, for twice the pairs.
//
// Slot s holds sorted atoms i0 = slot_atom[s] & 0x7fffffff and, unless bit 31
// is set, i1 = i0 + 1 (the same cell).  Its list uses the per-atom layout
// (groups of 32 slots, quads of entries; entry = (stencil << 27) | j, j never
// i0 or i1) and is padded to whole quads with entries that point at a far
// away dummy position stored after the last atom (index n).  The list is a
// superset of both atoms' lists: it accepts j when the float32 distance to
// either atom is below r_list^2 (1 + 2^-14), which covers every pair within
// r_list -- and so, by the half-skin rule, every pair within r_c until the
// next rebuild.  The force pass evaluates the slot's own pair once
// (f_i0 += F, f_i1 -= F), then both atoms against each list entry in
// float32 -- packed: one f32x2 instruction serves the two atoms -- with the
// per-atom kernel's velocity-Verlet epilogue.  Each atom's
// force is summed in float32 over the whole list (about 55 entries per atom
// at rho* = 0.8442, so one chunk of the per-atom kernel's float32-then-
// float64 sums) and converted once: without the float64 accumulators the
// kernel fits 8 CTAs of 128 threads per SM.
#include <algorithm>
#include <type_traits>

#include "k_pair.cuh"

namespace mdg {

namespace {

constexpr uint32_t kHomeStencil = 13;       // stencil cell (0, 0, 0)
constexpr int kPairBlock = 128;

__device__ __forceinline__ bool chain_off(const DevStatus *ds, bool gated) {
    return ds->status != 0 || (gated && ds->rebuild == 0);
}

// The union list of each slot: the 27 cells around the slot's cell, in stencil
// order, their atoms four at a time (CandGroup).  A candidate j is tested
// against both atoms at once from the slot's midpoint m = (x0 + x1) / 2 and half
// separation u = (x1 - x0) / 2: the nearer atom's squared distance is
// |x_j - m|^2 + |u|^2 - 2 |(x_j - m).u|, so with the record's |x_j|^2 the test
//     |x_j|^2 - 2 m.x_j + (|m|^2 + |u|^2 - hi) < |2 u.x_j - 2 u.m|
// is an addition and six multiply-adds -- packed, for two candidates at a time --
// and one comparison.  m is taken in the candidate's cell frame, so every term
// stays below about 24 r_list^2 (cells of up to 4/3 r_list), and the float32
// rounding below about 1e-5 r_list^2, against the margin of 6e-5 r_list^2 in hi =
// r_list^2 (1 + 2^-14): the list stays a superset of both atoms' r_list spheres.
//
// Accepted entries go to a queue of the thread in shared memory (a store and an
// addition, both predicated) and from there to the list in whole quads: writing
// them one by one took eight instructions per candidate, accepted or not, and a
// scattered 4-byte store.  Bound by the latency of the candidate loads (L1 wavefronts
// 72 %, issue 46 %); eight blocks per SM with 40 queue rows measured best.
// Binning and list, two distance products per candidate against this form: 4.73 ->
// 3.80 ms at 9.8 M porous atoms, 0.565 -> 0.461 at 1 M (liquid), 1.19 -> 0.94 for
// 2.4 M atoms in 64 boxes (binning included, itself shorter than before).  Six and
// seven blocks with the next group prefetched: 4.14 and 4.26 ms; nine blocks: 3.86.
// MULTI (a batch of boxes): each slot takes the geometry of its atoms' box
// (cells numbered box after box from the box's cell0).
constexpr int kListRows = 40;                 // queue entries per thread
constexpr int kListChunk = 7;                 // candidate groups between queue checks
constexpr int kListHigh = kListRows - 4 * kListChunk;  // a fuller queue is emptied first

template <bool WRITE, bool MULTI = false>
__global__ void __launch_bounds__(kPairBlock, 8)
pair_list_kernel(int n, Grid g, const Grid *__restrict__ grids, const uint16_t *__restrict__ rep,
                 float hi, const float4 *__restrict__ xq, const CandGroup *__restrict__ cand,
                 const int32_t *__restrict__ cell, const int32_t *__restrict__ start,
                 const int32_t *__restrict__ slot_start, const uint32_t *__restrict__ slot_atom,
                 uint32_t *__restrict__ list, int32_t *__restrict__ count, int cap, DevStatus *ds,
                 bool gated, bool close) {
    __shared__ uint32_t s_queue[WRITE ? kListRows : 1][kPairBlock];
    if (chain_off(ds, gated)) return;
    const int nslots = slot_start[g.ncells];
    if (blockIdx.x == 0 && threadIdx.x == 0) ds->pair_slots = nslots;
    unsigned long long tot = 0;
    int overflow = 0, maxc = 0;
    const uint32_t pad = (kHomeStencil << kIndexBits) | (uint32_t)n;
    uint32_t *const q0p = &s_queue[0][threadIdx.x];
    const int capq = cap >> 2;
    // grid-stride over whole warps, so every lane reaches the reductions below
    const int stride = gridDim.x * blockDim.x;
    const int send = ((nslots + 31) & ~31);
    for (int s = blockIdx.x * blockDim.x + threadIdx.x; s < send; s += stride) {
        const bool on = s < nslots;
        const uint32_t sa = slot_atom[on ? s : nslots - 1];
        const int i0 = (int)(sa & ~kSingle);
        const int i1 = (sa & kSingle) ? i0 : i0 + 1;
        float mx, my, mz, ux, uy, uz, lim;  // u doubled
        {
            const float4 q0 = xq[i0], q1 = xq[i1];
            ux = q1.x - q0.x;
            uy = q1.y - q0.y;
            uz = q1.z - q0.z;
            mx = q0.x + 0.5f * ux;
            my = q0.y + 0.5f * uy;
            mz = q0.z + 0.5f * uz;
            lim = 0.25f * (ux * ux + uy * uy + uz * uz) - hi;
        }
        int nx = g.nx, ny = g.ny, nz = g.nz, c0 = 0;
        float wx = g.wf[0], wy = g.wf[1], wz = g.wf[2];
        if (MULTI) {
            const Grid &gb = grids[rep[i0]];
            nx = gb.nx; ny = gb.ny; nz = gb.nz; c0 = gb.cell0;
            wx = gb.wf[0]; wy = gb.wf[1]; wz = gb.wf[2];
        }
        const int c = cell[i0] - c0;
        const int cx = c % nx, cy = (c / nx) % ny, cz = c / (nx * ny);
        uint4 *const row = reinterpret_cast<uint4 *>(list + list_group(s, cap)) + (s & 31);
        const uint32_t own0 = (kHomeStencil << kIndexBits) | (uint32_t)i0,
                       own1 = (kHomeStencil << kIndexBits) | (uint32_t)i1;
        uint32_t *qp = q0p;  // the queue's end
        int nq = 0;          // quads written
        int cnt = 0;         // entries (not WRITE)
        // whole quads of the queue to the list, the rest to its front
        auto empty = [&]() {
            const uint32_t *r = q0p;
            for (; qp - r >= 4 * kPairBlock; r += 4 * kPairBlock) {
                if (on && nq < capq)
                    row[(size_t)nq * 32] =
                        make_uint4(r[0], r[kPairBlock], r[2 * kPairBlock], r[3 * kPairBlock]);
                ++nq;
            }
            const int left = (int)(qp - r) / kPairBlock;
            if (left > 0) q0p[0] = r[0];
            if (left > 1) q0p[kPairBlock] = r[kPairBlock];
            if (left > 2) q0p[2 * kPairBlock] = r[2 * kPairBlock];
            qp = q0p + left * kPairBlock;
        };
        for (int dz = -1; dz <= 1; ++dz) {
            const int zz = cz + dz < 0 ? nz - 1 : (cz + dz == nz ? 0 : cz + dz);
            for (int dy = -1; dy <= 1; ++dy) {
                const int yy = cy + dy < 0 ? ny - 1 : (cy + dy == ny ? 0 : cy + dy);
                for (int dx = -1; dx <= 1; ++dx) {
                    const int xx = cx + dx < 0 ? nx - 1 : (cx + dx == nx ? 0 : cx + dx);
                    const int cn = c0 + (zz * ny + yy) * nx + xx;
                    const uint32_t st = (uint32_t)((dz + 1) * 9 + (dy + 1) * 3 + (dx + 1));
                    // the midpoint moved against the cell shift
                    const float sx = mx - (float)dx * wx, sy = my - (float)dy * wy,
                                sz = mz - (float)dz * wz;
                    const float2 mx2 = dup2(-2.f * sx), my2 = dup2(-2.f * sy), mz2 = dup2(-2.f * sz);
                    const float2 k1 = dup2(sx * sx + sy * sy + sz * sz + lim);
                    const float2 k2 = dup2(-(ux * sx + uy * sy + uz * sz));
                    const float2 ux2 = dup2(ux), uy2 = dup2(uy), uz2 = dup2(uz);
                    const int b = start[cn], e = start[cn + 1];
                    const CandGroup *gp = cand + cell_group0(cn, b);
                    const int ng = (e - b + 3) >> 2;
                    // every lane makes the warp's largest number of rounds, so that
                    // all of them vote together on emptying the queues
                    const int ngw = (int)__reduce_max_sync(0xffffffffu, (unsigned)ng);
                    uint32_t ent = (st << kIndexBits) | (uint32_t)b;
                    // HOME: the slot's own cell, the only one that holds i0 and i1
                    auto scan = [&](auto home) {
                        constexpr bool HOME = decltype(home)::value;
                        for (int g0 = 0; g0 < ngw; g0 += kListChunk) {
                            const int ge = min(ng, g0 + kListChunk);
                            for (int gi = g0; gi < ge; ++gi, ent += 4) {
                                const float4 X = __ldg(&gp[gi].x), Y = __ldg(&gp[gi].y),
                                             Z = __ldg(&gp[gi].z), W = __ldg(&gp[gi].w);
                                const float2 xa = make_float2(X.x, X.y), xb = make_float2(X.z, X.w);
                                const float2 ya = make_float2(Y.x, Y.y), yb = make_float2(Y.z, Y.w);
                                const float2 za = make_float2(Z.x, Z.y), zb = make_float2(Z.z, Z.w);
                                const float2 wa = make_float2(W.x, W.y), wb = make_float2(W.z, W.w);
                                const float2 ra = fma2(za, mz2, fma2(ya, my2, fma2(xa, mx2, add2(wa, k1))));
                                const float2 rb = fma2(zb, mz2, fma2(yb, my2, fma2(xb, mx2, add2(wb, k1))));
                                const float2 pa = fma2(za, uz2, fma2(ya, uy2, fma2(xa, ux2, k2)));
                                const float2 pb = fma2(zb, uz2, fma2(yb, uy2, fma2(xb, ux2, k2)));
                                auto take = [&](float r, float p, uint32_t en) {
                                    bool acc = r < fabsf(p);
                                    if (HOME) acc = acc & (en != own0) & (en != own1);
                                    if (WRITE) {
                                        if (acc) {
                                            *qp = en;
                                            qp += kPairBlock;
                                        }
                                    } else {
                                        cnt += acc ? 1 : 0;
                                    }
                                };
                                take(ra.x, pa.x, ent);
                                take(ra.y, pa.y, ent + 1);
                                take(rb.x, pb.x, ent + 2);
                                take(rb.y, pb.y, ent + 3);
                            }
                            if (WRITE && __any_sync(0xffffffffu, qp - q0p > kListHigh * kPairBlock))
                                empty();
                        }
                    };
                    if (st == kHomeStencil) scan(std::true_type{});
                    else scan(std::false_type{});
                }
            }
        }
        if (WRITE) {
            empty();
            const int left = (int)(qp - q0p) / kPairBlock;
            cnt = 4 * nq + left;
            if (on && left > 0 && nq < capq)
                row[(size_t)nq * 32] = make_uint4(q0p[0], left > 1 ? q0p[kPairBlock] : pad,
                                                  left > 2 ? q0p[2 * kPairBlock] : pad, pad);
            if (on) count[s] = cnt;
        }
        if (on) {
            maxc = max(maxc, cnt);
            tot += (unsigned long long)cnt;
            overflow |= (cnt > cap);
        }
    }
    for (int o = 16; o > 0; o >>= 1) tot += __shfl_down_sync(0xffffffffu, tot, o);
    maxc = (int)__reduce_max_sync(0xffffffffu, (unsigned)maxc);
    if ((threadIdx.x & 31) == 0) {
        if (tot) atomicAdd(&ds->pair_entries, tot);
        if (maxc) atomicMax(&ds->pair_max, maxc);
    }
    if (WRITE && overflow) atomicCAS(&ds->status, 0, (int)MD_ERR_LIST_OVERFLOW);
    list_build_done(ds, close);
}

// The same lists for small systems, a warp per slot (as warp_list_kernel): the
// lanes take a cell's candidates at once.  The test is the midpoint form
// |e|^2 - 2 |e.u| < hi - |u|^2 with e = x_j - m and u the half separation.
template <bool WRITE>
__global__ void __launch_bounds__(kPairBlock)
warp_pair_list_kernel(int n, Grid g1, const Grid *__restrict__ grids,
                      const uint16_t *__restrict__ rep, float hi, const float4 *__restrict__ xq,
                      const int32_t *__restrict__ cell, const int32_t *__restrict__ start,
                      const int32_t *__restrict__ slot_start,
                      const uint32_t *__restrict__ slot_atom, uint32_t *__restrict__ list,
                      int32_t *__restrict__ count, int cap, DevStatus *ds, bool gated, bool close) {
    if (chain_off(ds, gated)) return;
    const int nslots = slot_start[g1.ncells];
    if (blockIdx.x == 0 && threadIdx.x == 0) ds->pair_slots = nslots;
    const int lane = threadIdx.x & 31;
    const int nw = gridDim.x * (kPairBlock / 32);
    unsigned long long tot = 0;
    int overflow = 0, maxc = 0;
    for (int s = blockIdx.x * (kPairBlock / 32) + (threadIdx.x >> 5); s < nslots; s += nw) {
        const uint32_t sa = slot_atom[s];
        const int i0 = (int)(sa & ~kSingle);
        const int i1 = (sa & kSingle) ? i0 : i0 + 1;
        const Grid &g = grids[rep ? rep[i0] : 0];
        const float4 q0 = xq[i0], q1 = xq[i1];
        const float ux = 0.5f * (q1.x - q0.x), uy = 0.5f * (q1.y - q0.y), uz = 0.5f * (q1.z - q0.z);
        const float mx = q0.x + ux, my = q0.y + uy, mz = q0.z + uz;
        const float lim = hi - (ux * ux + uy * uy + uz * uz);
        const int c = cell[i0] - g.cell0;
        int b = 0, e = 0, dx, dy, dz;
        if (lane < kStencil) {
            const int cn = stencil_cell(g, c % g.nx, (c / g.nx) % g.ny, c / (g.nx * g.ny), lane, dx,
                                        dy, dz);
            b = start[cn];
            e = start[cn + 1];
        }
        uint32_t *row = list + list_group(s, cap) + ((s & 31) << 2);
        const float wx = g.wf[0], wy = g.wf[1], wz = g.wf[2];
        int cnt = 0;
#pragma unroll 3
        for (int st = 0; st < kStencil; ++st) {
            const int sb = __shfl_sync(0xffffffffu, b, st), se = __shfl_sync(0xffffffffu, e, st);
            const float sx = mx - (float)(st % 3 - 1) * wx, sy = my - (float)((st / 3) % 3 - 1) * wy,
                        sz = mz - (float)(st / 9 - 1) * wz;
            for (int j0 = sb; j0 < se; j0 += 32) {
                const int j = j0 + lane;
                bool acc = false;
                if (j < se) {
                    const float4 qj = xq[j];
                    const float ex = qj.x - sx, ey = qj.y - sy, ez = qj.z - sz;
                    const float r2 = ex * ex + ey * ey + ez * ez;
                    const float p = ex * ux + ey * uy + ez * uz;
                    acc = fmaf(-2.0f, fabsf(p), r2) < lim;
                    if (st == (int)kHomeStencil) acc = acc && j != i0 && j != i1;
                }
                const unsigned m = __ballot_sync(0xffffffffu, acc);
                if (WRITE && acc) {
                    const int k = cnt + __popc(m & ((1u << lane) - 1u));
                    if (k < cap) row[k + (k >> 2) * 124] = ((uint32_t)st << kIndexBits) | (uint32_t)j;
                }
                cnt += __popc(m);
            }
        }
        if (WRITE && cnt <= cap && lane < ((-cnt) & 3)) {
            const int k = cnt + lane;
            row[k + (k >> 2) * 124] = (kHomeStencil << kIndexBits) | (uint32_t)n;
        }
        if (lane == 0 && WRITE) count[s] = cnt;
        maxc = max(maxc, cnt);
        tot += (unsigned long long)cnt;
        overflow |= (cnt > cap);
    }
    if (lane == 0) {
        if (tot) atomicAdd(&ds->pair_entries, tot);
        if (maxc) atomicMax(&ds->pair_max, maxc);
        if (WRITE && overflow) atomicCAS(&ds->status, 0, (int)MD_ERR_LIST_OVERFLOW);
    }
    list_build_done(ds, close);
}

// the dummy neighbour of the padding entries, past the last atom of both
// position buffers and of the many-body passes' (x, F') records
__global__ void pair_dummy_kernel(float4 *xq0, float4 *xq1, float4 *xqf, int n) {
    const float4 far = make_float4(3.0e18f, 3.0e18f, 3.0e18f, 0.f);
    xq0[n] = far;
    xq1[n] = far;
    if (xqf) xqf[n] = far;
}

// Measured on GB300 (porous LJ, 9.8 M atoms, one force launch), with the cell
// shifts still read from a table: packed pairs and float32 sums at 56 registers
// 1.232 ms against 1.304 ms for the per-atom kernel from the generated state; the
// same arithmetic unpacked 1.387 ms (issue-bound: the second atom's pair terms
// cost as many instructions as the first's); with float64 chunk accumulators at
// 72 registers (7 CTAs) 1.498 ms unpacked and 1.551 ms packed (latency-bound).
// With the shifts computed (stencil_of), 9 / 8 / 7 CTAs per SM, whole runs: liquid
// of 1 M atoms 6.49 / 6.17 / 6.30 ms, 64 boxes 13.93 / 12.40 / 13.28
// (9 CTAs leave 56 registers a thread, 8 leave 64).  The persistent kernel, whose
// next tile is prefetched, keeps 9 (porous 9.8 M 64.6 / 65.0 / 66.6).
// MULTI: a batch of boxes.
//
// P > 1: thread t serves slot t / P.
template <int MODE, bool ENERGY, bool MULTI = false, int P = 1>
__global__ void __launch_bounds__(kPairBlock, P > 1 ? 1 : 8)
lj_pair_kernel(ForceArgs a, PairArgs p, int store_f) {
    if (a.ds->status != 0) return;
    step_bookkeeping<MODE>(a);
    const int nslots = p.slot_start[p.ncells];
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if constexpr (P > 1) {
        if ((t & ~31) / P >= nslots) return;  // whole warps: the lanes add their sums
        const bool on = t / P < nslots;
        lj_pair_slot<MODE, ENERGY, MULTI, P>(a, p, on ? t / P : nslots - 1, store_f, t % P, on);
    } else if (t < nslots) {
        lj_pair_slot<MODE, ENERGY, MULTI>(a, p, t, store_f);
    }
}

}  // namespace

int64_t pair_slots_max(int64_t n, int ncells) { return (n + ncells) / 2 + 1; }

cudaError_t launch_pair_dummy(md_system *h) {
    pair_dummy_kernel<<<1, 1, 0, h->stream>>>(h->xq[0], h->xq[1], h->xqf, (int)h->n);
    return cudaGetLastError();
}

cudaError_t launch_pair_build(md_system *h, bool write, bool gated, bool close) {
    const int n = (int)h->n, nc = h->g.ncells;
    cudaStream_t s = h->stream;
    if (!gated) {
        const cudaError_t e = launch_reset_counts(h, true);
        if (e != cudaSuccess) return e;
    }
    const int64_t smax = pair_slots_max(h->n, nc);
    if (h->n / 2 <= kWarpListItems) {
        const int nb = (int)((smax + kPairBlock / 32 - 1) / (kPairBlock / 32));
        auto k = write ? warp_pair_list_kernel<true> : warp_pair_list_kernel<false>;
        k<<<std::min(nb, 152 * 128), kPairBlock, 0, s>>>(n, h->g, h->grids, h->rep, h->list_hi,
                                                         h->xq[h->cur], h->cell, h->cell_start,
                                                         h->ps_start, h->ps_atom, h->ps_list,
                                                         h->ps_count, h->ps_cap, h->ds, gated, close);
        return cudaGetLastError();
    }
    const int blocks = (int)std::min<int64_t>((smax + kPairBlock - 1) / kPairBlock, 152 * 16);
#define MDG_PAIR_LIST(W, M)                                                                  \
    pair_list_kernel<W, M><<<blocks, kPairBlock, 0, s>>>(                                    \
        n, h->g, h->grids, h->rep, h->list_hi, h->xq[h->cur], h->cand, h->cell, h->cell_start,       \
        h->ps_start, h->ps_atom, h->ps_list, h->ps_count, h->ps_cap, h->ds, gated, close)
    if (h->R > 1) {
        if (write) MDG_PAIR_LIST(true, true);
        else MDG_PAIR_LIST(false, true);
    } else {
        if (write) MDG_PAIR_LIST(true, false);
        else MDG_PAIR_LIST(false, false);
    }
#undef MDG_PAIR_LIST
    return cudaGetLastError();
}

// the multi-element variant (k_pair_typed.cu)
cudaError_t launch_pair_typed_forces(md_system *h, int mode, bool energy, bool store_f);

template <bool MULTI, int P>
static cudaError_t launch_pair_lj(md_system *h, int mode, bool energy, int sf) {
    const ForceArgs a = make_force_args(h);
    const PairArgs p = make_pair_args(h);
    const int nb = pair_grid_blocks(h, kPairBlock, P);
    cudaStream_t s = h->stream;
    switch (mode) {
        case FM_STORE:
            if (energy) lj_pair_kernel<FM_STORE, true, MULTI, P><<<nb, kPairBlock, 0, s>>>(a, p, sf);
            else lj_pair_kernel<FM_STORE, false, MULTI, P><<<nb, kPairBlock, 0, s>>>(a, p, sf);
            break;
        case FM_FUSED_FULL:
            lj_pair_kernel<FM_FUSED_FULL, false, MULTI, P><<<nb, kPairBlock, 0, s>>>(a, p, sf);
            break;
        default: lj_pair_kernel<FM_FUSED_HALF, false, MULTI, P><<<nb, kPairBlock, 0, s>>>(a, p, sf); break;
    }
    return cudaGetLastError();
}

cudaError_t launch_pair_forces(md_system *h, int mode, bool energy, bool store_f) {
    if (h->fc.ntypes > 0) return launch_pair_typed_forces(h, mode, energy, store_f);
    const int sf = store_f ? 1 : 0;
    const int P = mixed_split(h->n / 2, h->ps_cap, kFourLanesSlots);
    if (h->R > 1)
        return P == 8 ? launch_pair_lj<true, 8>(h, mode, energy, sf)
             : P == 4 ? launch_pair_lj<true, 4>(h, mode, energy, sf)
                      : launch_pair_lj<true, 1>(h, mode, energy, sf);
    return P == 8 ? launch_pair_lj<false, 8>(h, mode, energy, sf)
         : P == 4 ? launch_pair_lj<false, 4>(h, mode, energy, sf)
                  : launch_pair_lj<false, 1>(h, mode, energy, sf);
}

}  // namespace mdg
