// k_bin.cu -- cell binning by counting sort (Sec. 2.1: the volume is divided
// into small cells; a cell's atoms are processed together).
//
// Atoms are assigned to cell c = min(floor(x * n_d / L_d), n_d - 1) per
// dimension, counted with atomics, the counts are scanned into cell starts and
// atoms are scattered into their cell's range.  One warp per cell then orders
// the cell's atoms -- by original id, so that the sorted layout is
// deterministic and equals a stable sort by (cell, original id), or, for the
// two-atom layout, whose slots take a cell's atoms two at a time, in a pairing
// order (also deterministic) that places near neighbours next to each other --
// and gathers the state in that order as float64 positions relative to the
// cell centre plus their float32 copy (the layout the force kernels read).
//
// Traffic: the counting pass also writes each atom's absolute position and
// velocity (with its original id, new cell and replica packed into the spare
// fourth words) into two 32-byte records, so the gather reads two aligned
// sectors per atom instead of seven scattered words.
//
// Launches: five (counting, two of the scan, scatter, order and gather); the
// slot tables of the two-atom layout come out of the scan (slots per cell, beside
// the atoms) and of the last pass.  Every step holds the gated chain, and an idle
// kernel of it costs 0.5 us in a replayed step (2 us where the steps are launched
// one by one), so the chain is kept short: with the list build six launches, where
// passes of their own (zeroing, sorting, gathering, slot tables, closing) made
// eleven, eighteen under the two-atom layout.  The records are read once: 40 steps
// of 9.8 M porous atoms went from 69.7 to 68.6 ms.
//
// A system of several boxes (replicas) numbers its cells consecutively, box
// after box, so each box's atoms stay one contiguous range of the sorted
// order; every kernel reads the geometry of the atom's own box.
#include "k_scan.cuh"

#include <algorithm>
#include <climits>

namespace mdg {

namespace {

__device__ __forceinline__ bool chain_off(const DevStatus *ds, bool gated) {
    return ds->status != 0 || (gated && ds->rebuild == 0);
}

// floor(x * inv_w) clamped to [0, n-1] (one float64 floor-convert: the
// conversion saturates, and a NaN coordinate converts to 0, so an exploding
// state can never index outside the cell arrays; the drift check reports it
// as MD_ERR_NONFINITE).
__device__ __forceinline__ int cell_coord(double x, double inv_w, int n) {
    const int q = __double2int_rd(x * inv_w);
    return q < 0 ? 0 : (q > n - 1 ? n - 1 : q);
}

// Absolute position of sorted atom i: exact in xabs right after a build or a
// load (abs_fresh); otherwise the cell centre plus the relative position.  An
// atom of an interior cell whose offset is below the cell width lies strictly
// inside the box, so only boundary cells and stray offsets need the periodic
// wrap.  cell < 0: xr holds the absolute position (a loaded state).
__device__ __forceinline__ double3 absolute_position(int i, const Grid &g, bool fresh,
                                                     const double4 *__restrict__ xr,
                                                     const int32_t *__restrict__ cell,
                                                     const double4 *__restrict__ xabs) {
    if (fresh) {
        const double4 a = xabs[i];
        return make_double3(a.x, a.y, a.z);
    }
    const double4 r = xr[i];
    const int c = cell[i];
    double x = r.x, y = r.y, z = r.z;
    if (c >= 0) {
        const int cl = c - g.cell0;
        const int cx = cl % g.nx, cy = (cl / g.nx) % g.ny, cz = cl / (g.nx * g.ny);
        const double3 C = cell_centre_of(cx, cy, cz, g);
        x = C.x + x; y = C.y + y; z = C.z + z;
        if (cx == 0 || cx == g.nx - 1 || !below_cell_width(r.x, g)) x = wrap_coord(x, g.L[0]);
        if (cy == 0 || cy == g.ny - 1 || !below_cell_width(r.y, g)) y = wrap_coord(y, g.L[1]);
        if (cz == 0 || cz == g.nz - 1 || !below_cell_width(r.z, g)) z = wrap_coord(z, g.L[2]);
    } else {
        x = wrap_coord(x, g.L[0]); y = wrap_coord(y, g.L[1]); z = wrap_coord(z, g.L[2]);
    }
    return make_double3(x, y, z);
}

// Spare fourth words of the gather records: (new cell << 32 | original id)
// beside the position, the replica beside the velocity.
__device__ __forceinline__ double pack2(int hi, int lo) {
    return __longlong_as_double(((long long)hi << 32) | (long long)(unsigned)lo);
}

// Cell of every atom, its slot in the cell (atomic count) and its gather
// records: (x, y, z, new cell | original id) and (v, replica).  The counts are
// zero on entry (the scan clears them behind itself).  Resets what the later
// passes of the rebuild count (not the list's counts when no list build follows:
// the last list's stay).
__global__ void bin_count_kernel(int n, const Grid *__restrict__ grids,
                                 const uint16_t *__restrict__ rep,
                                 const double4 *__restrict__ xr,
                                 const int32_t *__restrict__ cell,
                                 const double4 *__restrict__ xabs,
                                 const double *__restrict__ v, const int32_t *__restrict__ orig,
                                 int32_t *__restrict__ count, int32_t *__restrict__ new_cell,
                                 int32_t *__restrict__ slot, double4 *__restrict__ tabs,
                                 double4 *__restrict__ tv, bool slots, bool list_follows,
                                 DevStatus *ds, bool gated, bool count_run) {
    if (chain_off(ds, gated)) return;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        if (count_run) ds->cond_runs += 1;
        ds->max_cell = 0;
        if (list_follows) reset_list_counts(ds, slots);
    }
    const bool fresh = ds->abs_fresh != 0;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const int r = rep ? rep[i] : 0;
        const Grid &g = grids[r];
        const double3 x = absolute_position(i, g, fresh, xr, cell, xabs);
        const int cx = cell_coord(x.x, g.inv_w[0], g.nx);
        const int cy = cell_coord(x.y, g.inv_w[1], g.ny);
        const int cz = cell_coord(x.z, g.inv_w[2], g.nz);
        const int c = g.cell0 + (cz * g.ny + cy) * g.nx + cx;
        new_cell[i] = c;
        slot[i] = atomicAdd(&count[c], 1);
        tabs[i] = make_double4(x.x, x.y, x.z, pack2(c, orig[i]));
        tv[i] = make_double4(v[i], v[n + i], v[2 * (size_t)n + i], pack2(0, r));
    }
}

// Exclusive prefix sums over the cells of the atoms and of the slots
// (ceil(atoms / 2)) of every cell at once, the two sums packed in one 64-bit
// word (slots << 32 | atoms, each below 2^31); the counts are cleared behind the
// read, and the largest cell is noted.  slot_start may be null.
__global__ void __launch_bounds__(kBlock)
cell_scan_block_kernel(int32_t *__restrict__ count, int32_t *__restrict__ start,
                       int32_t *__restrict__ slot_start, int n, long long *__restrict__ bsum,
                       DevStatus *ds, bool gated) {
    if (chain_off(ds, gated)) return;
    __shared__ long long tot;
    const long long base = (long long)blockIdx.x * kScanTile + (long long)threadIdx.x * kScanItems;
    int c[kScanItems];
    long long s = 0;
    int maxc = 0;
#pragma unroll
    for (int k = 0; k < kScanItems; ++k) {
        const long long idx = base + k;
        c[k] = 0;
        if (idx < n) {
            c[k] = count[idx];
            count[idx] = 0;
        }
        maxc = max(maxc, c[k]);
        s += ((long long)((c[k] + 1) >> 1) << 32) + c[k];
    }
    long long off = block_exclusive<long long>(s, &tot);
#pragma unroll
    for (int k = 0; k < kScanItems; ++k) {
        const long long idx = base + k;
        if (idx < n) {
            start[idx] = (int)(unsigned)off;
            if (slot_start) slot_start[idx] = (int)(off >> 32);
        }
        off += ((long long)((c[k] + 1) >> 1) << 32) + c[k];
    }
    if (threadIdx.x == 0) bsum[blockIdx.x] = tot;
    maxc = (int)__reduce_max_sync(0xffffffffu, (unsigned)maxc);
    if ((threadIdx.x & 31) == 0 && maxc) atomicMax(&ds->max_cell, maxc);
}

// adds the tiles before (one block per tile; as scan_add_kernel)
__global__ void __launch_bounds__(kBlock)
cell_scan_add_kernel(int32_t *__restrict__ start, int32_t *__restrict__ slot_start, int n,
                     const long long *__restrict__ bsum, int nb, bool prefixed,
                     const DevStatus *ds, bool gated) {
    if (chain_off(ds, gated)) return;
    const int t = blockIdx.x;
    const long long off = prefixed ? bsum[t] : tiles_before<long long>(bsum, t);
    const long long b = (long long)t * kScanTile;
#pragma unroll
    for (int k = 0; k < kScanItems; ++k) {
        const long long idx = b + (long long)k * kBlock + threadIdx.x;
        if (idx < n) {
            start[idx] += (int)(unsigned)off;
            if (slot_start) slot_start[idx] += (int)(off >> 32);
        }
    }
    if (t == nb - 1 && threadIdx.x == 0) {
        const long long end = prefixed ? bsum[nb] : off + bsum[t];
        start[n] = (int)(unsigned)end;
        if (slot_start) slot_start[n] = (int)(end >> 32);
    }
}

__global__ void scatter_kernel(int n, const int32_t *__restrict__ new_cell,
                               const int32_t *__restrict__ slot,
                               const int32_t *__restrict__ start, int32_t *__restrict__ src,
                               const DevStatus *ds, bool gated) {
    if (chain_off(ds, gated)) return;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
        src[start[new_cell[i]] + slot[i]] = i;
}

// What the last pass writes, in the new order.
struct GatherArgs {
    int n;
    const Grid *grids;
    const double4 *tabs, *tv;  // the counting pass's records
    double4 *xr;
    float4 *xq, *xq_build;
    double4 *xabs;
    double *v;
    int32_t *orig, *cell;
    uint16_t *rep;
    const int32_t *type_orig;
    CandGroup *cand;  // null: not the two-atom layout
};

__device__ __forceinline__ int record_orig(const double4 &a) {
    return (int)(unsigned)(__double_as_longlong(a.w) & 0xffffffffll);
}

// the atom of record s (position record a) becomes sorted atom k of the cell whose
// range starts at b
__device__ __forceinline__ void gather_atom(const GatherArgs &o, int b, int k, int s,
                                            const double4 &a) {
    const double4 u = o.tv[s];
    const int id = record_orig(a);
    const int c = (int)(__double_as_longlong(a.w) >> 32);
    const int r = (int)(__double_as_longlong(u.w) & 0xffff);
    const Grid &g = o.grids[r];
    const int cl = c - g.cell0;
    const double3 C = cell_centre_of(cl % g.nx, (cl / g.nx) % g.ny, cl / (g.nx * g.ny), g);
    const double rx = a.x - C.x, ry = a.y - C.y, rz = a.z - C.z;
    o.xr[k] = make_double4(rx, ry, rz, 0.0);
    // the float32 word carries the original id and, for a multi-element
    // system, the species above it
    const uint32_t w = (uint32_t)id | (o.type_orig ? (uint32_t)o.type_orig[id] << kIndexBits : 0u);
    const float4 q = make_float4((float)rx, (float)ry, (float)rz, __uint_as_float(w));
    o.xq[k] = q;
    o.xq_build[k] = q;
    if (o.cand) {
        float *g4 =
            reinterpret_cast<float *>(o.cand + cell_group0(c, b) + ((k - b) >> 2)) + ((k - b) & 3);
        g4[0] = q.x;
        g4[4] = q.y;
        g4[8] = q.z;
        g4[12] = q.x * q.x + q.y * q.y + q.z * q.z;
    }
    o.xabs[k] = make_double4(a.x, a.y, a.z, 0.0);
    const size_t n = (size_t)o.n;
    o.v[k] = u.x;
    o.v[n + k] = u.y;
    o.v[2 * n + k] = u.z;
    o.orig[k] = id;
    o.cell[k] = c;
    if (o.rep) o.rep[k] = (uint16_t)r;
}

// A cell by original id, any occupancy, by its warp: the rank of an atom is the
// number of smaller ids in the cell (they are distinct).  Up to 32 atoms by
// shuffles; above that each lane ranks every 32nd atom by reading the cell's
// ids (uniform, independent reads).
constexpr int kOrderBlock = 256;

__device__ __forceinline__ void gather_by_id(const GatherArgs &o, int b, int m, int lane,
                                             const int32_t *__restrict__ src) {
    if (m <= 32) {
        const int s = lane < m ? src[b + lane] : 0;
        const double4 a = lane < m ? o.tabs[s] : make_double4(0.0, 0.0, 0.0, 0.0);
        const int id = lane < m ? record_orig(a) : 0x7fffffff;
        int rank = 0;
        for (int q = 0; q < m; ++q) rank += (__shfl_sync(0xffffffffu, id, q) < id) ? 1 : 0;
        if (lane < m) gather_atom(o, b, b + rank, s, a);
        return;
    }
    for (int l = lane; l < m; l += 32) {
        const int s = src[b + l];
        const double4 a = o.tabs[s];
        const int id = record_orig(a);
        int rank = 0;
#pragma unroll 4
        for (int q = 0; q < m; ++q)
            rank += (int)(unsigned)(__double_as_longlong(o.tabs[src[b + q]].w) & 0xffffffffll) < id ? 1 : 0;
        gather_atom(o, b, b + rank, s, a);
    }
}

// the empty places of a cell's last candidate group
__device__ __forceinline__ void pad_group(const GatherArgs &o, int c, int b, int m, int lane) {
    if (lane < ((-m) & 3)) {
        const int k = m + lane;
        float *g4 = reinterpret_cast<float *>(o.cand + cell_group0(c, b) + (k >> 2)) + (k & 3);
        g4[0] = g4[4] = g4[8] = 0.f;
        g4[12] = __int_as_float(0x7f800000);
    }
}

// slots of a cell: first atoms, the last one flagged when it holds one atom
__device__ __forceinline__ void write_slots(int b, int m, int lane, int s0,
                                            uint32_t *__restrict__ slot_atom) {
    for (int k = lane; 2 * k < m; k += 32)
        slot_atom[s0 + k] = (uint32_t)(b + 2 * k) | (2 * k + 1 >= m ? 0x80000000u : 0u);
}

__global__ void __launch_bounds__(kOrderBlock)
cell_id_order_kernel(int ncells, const int32_t *__restrict__ start,
                     const int32_t *__restrict__ src, GatherArgs o, DevStatus *ds, bool gated) {
    if (chain_off(ds, gated)) return;
    if (blockIdx.x == 0 && threadIdx.x == 0) ds->abs_fresh = 1;
    const int lane = threadIdx.x & 31;
    const int nw = gridDim.x * (kOrderBlock / 32);
    for (int c = blockIdx.x * (kOrderBlock / 32) + (threadIdx.x >> 5); c < ncells; c += nw) {
        const int b = start[c], m = start[c + 1] - b;
        if (m > 0) gather_by_id(o, b, m, lane, src);
    }
}

// three bits per axis interleaved (x lowest): the octree position of a point
// in its cell at 1/8 of the cell width
__device__ __forceinline__ unsigned morton9(unsigned qx, unsigned qy, unsigned qz) {
    auto spread = [](unsigned v) { return (v & 1u) | ((v & 2u) << 2) | ((v & 4u) << 4); };
    return spread(qx) | (spread(qy) << 1) | (spread(qz) << 2);
}

// the octree coordinate, from float32 position and inverse width (products
// and differences rounded one by one)
__device__ __forceinline__ unsigned octree_coord(float x, float inv_w) {
    const float t = __fmul_rn(x, inv_w);
    const int q = (int)__fmul_rn(__fsub_rn(t, floorf(t)), 8.0f);
    return (unsigned)min(max(q, 0), 7);
}

// float64 to float32 rounded toward zero, from the IEEE-754 fields with
// integer operations (the float64 pipe is slow on this part); a value below
// the float32 normal range, zero included, gives 0
__device__ __forceinline__ float f32_toward_zero(double d) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(d);
    const unsigned hi = (unsigned)(b >> 32), lo = (unsigned)b;
    const int e = (int)((hi >> 20) & 0x7ffu) - 1023 + 127;
    const unsigned m = ((hi & 0xfffffu) << 3) | (lo >> 29);
    return e <= 0 ? 0.0f : __uint_as_float((hi & 0x80000000u) | ((unsigned)e << 23) | m);
}

// Pairing order for the two-atom layout, whose slot k of a cell holds the
// cell's sorted atoms 2k and 2k + 1: the union of two cut-off spheres grows
// with the distance between their centres, and a warp's loop runs as long as
// its longest slot list, so the pairs should be near neighbours.  One warp
// per cell of up to 32 atoms: the atoms are ranked by the Morton code of
// their octree position in the cell (ties by original id) and moved to the
// lane of their rank; then, while two or more are left, the first unpaired
// atom in rank takes the nearest unpaired atom (squared distance with its low
// 5 bits replaced by the rank, so ties go to the lower rank), and the two
// fill the next two places.  A cell of odd occupancy ends with the atom left
// over.  Positions are float32 (rounded toward zero from float64) and every
// product and sum is rounded on its own, so the order depends on positions
// and ids only and is deterministic; a larger cell falls back to the
// original-id order (cell_pair_order2_kernel is the form for systems whose
// average cell is larger).
__global__ void __launch_bounds__(kOrderBlock)
cell_pair_order_kernel(int ncells, const int32_t *__restrict__ start,
                       const int32_t *__restrict__ slot_start, uint32_t *__restrict__ slot_atom,
                       const int32_t *__restrict__ src, GatherArgs out, DevStatus *ds,
                       bool gated) {
    if (chain_off(ds, gated)) return;
    if (blockIdx.x == 0 && threadIdx.x == 0) ds->abs_fresh = 1;
    constexpr unsigned full = 0xffffffffu;
    __shared__ int s_lane_of[kOrderBlock / 32][32];
    int *lane_of = s_lane_of[threadIdx.x >> 5];
    const int lane = threadIdx.x & 31;
    const int nw = gridDim.x * (kOrderBlock / 32);
    for (int c = blockIdx.x * (kOrderBlock / 32) + (threadIdx.x >> 5); c < ncells; c += nw) {
        const int b = start[c], m = start[c + 1] - b;
        if (m == 0) continue;
        write_slots(b, m, lane, slot_start[c], slot_atom);
        pad_group(out, c, b, m, lane);
        if (m == 1 || m > 32) {
            gather_by_id(out, b, m, lane, src);
            continue;
        }
        const bool on = lane < m;
        int sv = on ? src[b + lane] : 0;
        const double4 a = on ? out.tabs[sv] : make_double4(0.0, 0.0, 0.0, 0.0);
        const int o = on ? record_orig(a) : 0x7fffffff;
        float px = f32_toward_zero(a.x), py = f32_toward_zero(a.y), pz = f32_toward_zero(a.z);
        // the cell's box (a cell's atoms share it)
        const Grid &g =
            out.grids[out.rep ? (int)(__double_as_longlong(out.tv[src[b]].w) & 0xffff) : 0];
        const float iwx = g.inv_wf[0], iwy = g.inv_wf[1], iwz = g.inv_wf[2];
        const unsigned mk =
            morton9(octree_coord(px, iwx), octree_coord(py, iwy), octree_coord(pz, iwz));
        const long long K = on ? (((long long)mk << 32) | (long long)o) : LLONG_MAX;
        int rank = 0;
        for (int q = 0; q < m; ++q) rank += (__shfl_sync(full, K, q) < K) ? 1 : 0;
        // lane r takes the atom of rank r
        if (on) lane_of[rank] = lane;
        __syncwarp();
        const int from = on ? lane_of[lane] : lane;
        __syncwarp();
        sv = __shfl_sync(full, sv, from);
        px = __shfl_sync(full, px, from);
        py = __shfl_sync(full, py, from);
        pz = __shfl_sync(full, pz, from);
        unsigned left = (m == 32) ? full : ((1u << m) - 1u);
        int dst = 0, next = 0;
        while (__popc(left) >= 2) {
            const int first = __ffs(left) - 1;
            const float fx = __shfl_sync(full, px, first), fy = __shfl_sync(full, py, first),
                        fz = __shfl_sync(full, pz, first);
            // atoms of one cell need no periodic image
            const float dx = __fsub_rn(px, fx), dy = __fsub_rn(py, fy), dz = __fsub_rn(pz, fz);
            const float d2 =
                __fadd_rn(__fadd_rn(__fmul_rn(dx, dx), __fmul_rn(dy, dy)), __fmul_rn(dz, dz));
            const bool cand = ((left >> lane) & 1u) && lane != first;
            const unsigned k2 = cand ? ((__float_as_uint(d2) & ~31u) | (unsigned)lane) : full;
            const int mate = (int)(__reduce_min_sync(full, k2) & 31u);
            if (lane == first) dst = next;
            if (lane == mate) dst = next + 1;
            next += 2;
            left &= ~((1u << first) | (1u << mate));
        }
        if ((left >> lane) & 1u) dst = next;
        if (on) gather_atom(out, b, b + dst, sv, out.tabs[sv]);
    }
}

// The same order for cells of up to 64 atoms, two per lane: for systems whose
// average cell holds more than 32 atoms (Sutton-Chen at r_list = 2.2 a has 43)
// and at most 52, so that nearly every cell fits.  The ranked atoms sit in
// shared memory; rank r belongs to lane r % 32.  Distances keep all but their
// low 6 bits.  Latency-bound (a chain of warp reductions per pair), hidden by
// 16 resident blocks of four warps.  Sutton-Chen, 1,048,576 atoms, 50 steps
// and six builds: 40.4 -> 34.8 ms against insertion-sorted cells in original-id
// order (that order pass alone took 0.27 ms per build).
constexpr int kWideCell = 64, kWideMean = 52;
constexpr int kWideBlock = 128;

__global__ void __launch_bounds__(kWideBlock)
cell_pair_order2_kernel(int ncells, const int32_t *__restrict__ start,
                        const int32_t *__restrict__ slot_start, uint32_t *__restrict__ slot_atom,
                        const int32_t *__restrict__ src, GatherArgs out, DevStatus *ds,
                        bool gated) {
    if (chain_off(ds, gated)) return;
    if (blockIdx.x == 0 && threadIdx.x == 0) ds->abs_fresh = 1;
    constexpr unsigned full = 0xffffffffu;
    __shared__ long long s_key[kWideBlock / 32][kWideCell];
    __shared__ float4 s_atom[kWideBlock / 32][kWideCell];  // by rank: position, source record
    long long *wkey = s_key[threadIdx.x >> 5];
    float4 *watom = s_atom[threadIdx.x >> 5];
    const int lane = threadIdx.x & 31;
    const int nw = gridDim.x * (kWideBlock / 32);
    for (int c = blockIdx.x * (kWideBlock / 32) + (threadIdx.x >> 5); c < ncells; c += nw) {
        const int b = start[c], m = start[c + 1] - b;
        if (m == 0) continue;
        write_slots(b, m, lane, slot_start[c], slot_atom);
        pad_group(out, c, b, m, lane);
        if (m == 1 || m > kWideCell) {
            gather_by_id(out, b, m, lane, src);
            continue;
        }
        float4 at[2];
        long long K[2];
        // the cell's box (its atoms share it)
        const Grid &g =
            out.grids[out.rep ? (int)(__double_as_longlong(out.tv[src[b]].w) & 0xffff) : 0];
#pragma unroll
        for (int t = 0; t < 2; ++t) {
            const int l = lane + 32 * t;
            const bool on = l < m;
            const int sv = on ? src[b + l] : 0;
            const double4 a = on ? out.tabs[sv] : make_double4(0.0, 0.0, 0.0, 0.0);
            const int o = on ? record_orig(a) : 0x7fffffff;
            at[t] = make_float4(f32_toward_zero(a.x), f32_toward_zero(a.y), f32_toward_zero(a.z),
                                __int_as_float(sv));
            const unsigned mk = morton9(octree_coord(at[t].x, g.inv_wf[0]),
                                        octree_coord(at[t].y, g.inv_wf[1]),
                                        octree_coord(at[t].z, g.inv_wf[2]));
            K[t] = on ? (((long long)mk << 32) | (long long)o) : LLONG_MAX;
            wkey[l] = K[t];
        }
        __syncwarp();
        int rank[2] = {0, 0};
        for (int q = 0; q < m; ++q) {
            const long long kq = wkey[q];
            rank[0] += kq < K[0] ? 1 : 0;
            rank[1] += kq < K[1] ? 1 : 0;
        }
#pragma unroll
        for (int t = 0; t < 2; ++t)
            if (lane + 32 * t < m) watom[rank[t]] = at[t];
        __syncwarp();
        const float4 a0 = lane < m ? watom[lane] : make_float4(0.f, 0.f, 0.f, 0.f);
        const float4 a1 = lane + 32 < m ? watom[lane + 32] : make_float4(0.f, 0.f, 0.f, 0.f);
        unsigned long long left = (m == 64) ? ~0ull : ((1ull << m) - 1ull);
        int dst0 = 0, dst1 = 0, next = 0;
        auto key_of = [&](const float4 &a, const float4 &f, int r, bool cand) -> unsigned {
            const float dx = __fsub_rn(a.x, f.x), dy = __fsub_rn(a.y, f.y),
                        dz = __fsub_rn(a.z, f.z);
            const float d2 =
                __fadd_rn(__fadd_rn(__fmul_rn(dx, dx), __fmul_rn(dy, dy)), __fmul_rn(dz, dz));
            return cand ? ((__float_as_uint(d2) & ~63u) | (unsigned)r) : full;
        };
        while (__popcll(left) >= 2) {
            const int first = __ffsll((long long)left) - 1;
            const float4 f = watom[first];
            const unsigned k0 = key_of(a0, f, lane, ((left >> lane) & 1ull) && lane != first);
            const unsigned k1 =
                key_of(a1, f, lane + 32, ((left >> (lane + 32)) & 1ull) && lane + 32 != first);
            const int mate = (int)(__reduce_min_sync(full, min(k0, k1)) & 63u);
            if (lane == first) dst0 = next;
            if (lane + 32 == first) dst1 = next;
            if (lane == mate) dst0 = next + 1;
            if (lane + 32 == mate) dst1 = next + 1;
            next += 2;
            left &= ~((1ull << first) | (1ull << mate));
        }
        if ((left >> lane) & 1ull) dst0 = next;
        if ((left >> (lane + 32)) & 1ull) dst1 = next;
        if (lane < m) {
            const int sv = __float_as_int(a0.w);
            gather_atom(out, b, b + dst0, sv, out.tabs[sv]);
        }
        if (lane + 32 < m) {
            const int sv = __float_as_int(a1.w);
            gather_atom(out, b, b + dst1, sv, out.tabs[sv]);
        }
        __syncwarp();  // the shared rows are rewritten by the warp's next cell
    }
}

__global__ void export_cells_kernel(int n, int ncells, const int32_t *__restrict__ orig,
                                    const int32_t *__restrict__ cell,
                                    const int32_t *__restrict__ start, int32_t *cell_of_atom,
                                    int64_t *cell_start) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n && cell_of_atom) cell_of_atom[orig[i]] = cell[i];
    if (i <= ncells && cell_start) cell_start[i] = start[i];
}

}  // namespace

cudaError_t launch_scan_i32(const int32_t *in, int32_t *out, int n, int32_t *bsum,
                            const DevStatus *ds, bool gated, cudaStream_t s) {
    return launch_scan<int32_t>(in, out, n, bsum, ds, gated, s);
}

cudaError_t launch_bin(md_system *h, bool gated, bool count_run, bool list_follows) {
    const int n = (int)h->n, nc = h->g.ncells;
    cudaStream_t s = h->stream;
    const int cur = h->cur;
    // (a variant switch that failed half-way may have left no slot tables)
    const bool paired = h->p.force_variant == MD_FORCE_PAIRED && h->ps_count != nullptr;
    bin_count_kernel<<<gs_blocks(n), kBlock, 0, s>>>(n, h->grids, h->rep, h->xr64[cur], h->cell,
                                                     h->xabs, h->v, h->orig, h->cell_count,
                                                     h->new_cell, h->slot, h->tmp_abs, h->tmp_v,
                                                     paired, list_follows, h->ds, gated,
                                                     count_run);
    int32_t *slot_start = paired ? h->ps_start : nullptr;
    const int nb = std::max((nc + kScanTile - 1) / kScanTile, 1);
    const bool prefixed = nb > kScanDirect;
    cell_scan_block_kernel<<<nb, kBlock, 0, s>>>(h->cell_count, h->cell_start, slot_start, nc,
                                                 h->cell_bsum, h->ds, gated);
    if (prefixed) scan_bsum_kernel<long long><<<1, kBlock, 0, s>>>(h->cell_bsum, nb, h->ds, gated);
    cell_scan_add_kernel<<<nb, kBlock, 0, s>>>(h->cell_start, slot_start, nc, h->cell_bsum, nb,
                                               prefixed, h->ds, gated);
    scatter_kernel<<<gs_blocks(n), kBlock, 0, s>>>(n, h->new_cell, h->slot, h->cell_start, h->src,
                                                   h->ds, gated);
    GatherArgs o;
    o.n = n;
    o.grids = h->grids;
    o.tabs = h->tmp_abs;
    o.tv = h->tmp_v;
    o.xr = h->xr64[cur];
    o.xq = h->xq[cur];
    o.xq_build = h->xq_build;
    o.xabs = h->xabs;
    o.v = h->v;
    o.orig = h->orig;
    o.cell = h->cell;
    o.rep = h->rep;
    o.type_orig = h->type_orig;
    o.cand = paired ? h->cand : nullptr;
    const int warps = kOrderBlock / 32;
    const int blocks = std::max(std::min((nc + warps - 1) / warps, kGridCap * 2), 1);
    // one atom per lane while the average cell fits a warp, two per lane above
    if (paired && h->n > 32 * (int64_t)nc && h->n <= kWideMean * (int64_t)nc)
        cell_pair_order2_kernel<<<std::max(std::min((nc + 3) / 4, kGridCap * 2), 1), kWideBlock, 0,
                                  s>>>(nc, h->cell_start, h->ps_start, h->ps_atom, h->src, o,
                                       h->ds, gated);
    else if (paired)
        cell_pair_order_kernel<<<blocks, kOrderBlock, 0, s>>>(
            nc, h->cell_start, h->ps_start, h->ps_atom, h->src, o, h->ds, gated);
    else
        cell_id_order_kernel<<<blocks, kOrderBlock, 0, s>>>(nc, h->cell_start, h->src, o, h->ds,
                                                           gated);
    return cudaGetLastError();
}

int scan_launch_count(long long n) { return scan_launches(n); }
int bin_launches(const md_system *h) { return 3 + scan_launches(h->g.ncells); }

cudaError_t launch_export_cells(md_system *h, int32_t *cell_of_atom, int64_t *cell_start) {
    int m = (int)(h->n > h->g.ncells + 1 ? h->n : h->g.ncells + 1);
    export_cells_kernel<<<nblocks(m), kBlock, 0, h->stream>>>(
        (int)h->n, h->g.ncells, h->orig, h->cell, h->cell_start, cell_of_atom, cell_start);
    return cudaGetLastError();
}

}  // namespace mdg
