// k_rebuild.cu -- particle binning, counting sort by cell and Verlet-list build.
//
// Sec. 3 (Code structure): Verlet neighbour lists are built efficiently from
// a spatial decomposition of the particles ("particle binning"); Sec. 5
// (Truncated Force Performance Study): the list update is ~30 % of the run
// time.  A rebuild of replica r runs only when rep_needs_rebuild(r) (the skin
// rule: some particle moved more than skin/2 since the last build, or the
// host forced it); every kernel here tests that flag per work item, so the
// whole sequence can sit in a CUDA graph and cost one early exit per kernel
// when no replica needs it.
//
// Sequence: k_bin (new cell of every particle, counts) -> k_scan
// (exclusive scan of the counts per replica) -> k_scatter (slot
// per particle) -> k_sortgather (order inside each cell by FP32 z offset,
// ties by user index, so the layout is a deterministic function of the
// positions; gather into the sorted arrays) -> k_nlist (27-cell search,
// each neighbour cell narrowed to its candidates within reach along z).
// Each stage is a device function; k_rebuild_cluster runs those up to the
// gather in one launch for small boxes.
#include <climits>

#include "ljmd_internal.cuh"

namespace {

constexpr int kScanThreads = 256;
constexpr int kScanTile = 2048;   // cells per scan tile
// The cluster rebuild: one cluster of 16 blocks (the most a cluster may hold)
constexpr int kClusterBlocks = 16;
constexpr int kClusterThreads = 512;

__device__ __forceinline__ int cell_coords(const RepDev& R, int gc, int& cx, int& cy)
{
    int local = gc - R.cell_off;
    cx = local % R.nc[0];
    int t = local / R.nc[0];
    cy = t % R.nc[1];
    return t / R.nc[1];
}

// How many there are, of chunks and of cells (one replica: all of its own).
__device__ __forceinline__ int work_chunks(const BoxDev& b) { return b.nrep == 1 ? b.nchunk : b.lw_coff[b.lw_hdr[0]]; }
__device__ __forceinline__ int work_cells(const BoxDev& b) { return b.nrep == 1 ? b.ncell : b.lw_off[b.lw_hdr[0]]; }

// Cell (chunk) t of the concatenation of the rebuilding replicas' cells
// (particle chunks), from k_list_work's lists; kr is the replica index of the
// caller's previous t (t only grows).  Found by bisection: a block's first t
// lies behind up to all of the rebuilding replicas (~50 of 512 a step: 615 ->
// 610 us a step against a walk).
__device__ __forceinline__ int work_replica(const BoxDev& b, const int* off, int t, int kr)
{
    if (t < off[kr + 1]) return kr;
    int lo = kr + 1, hi = b.lw_hdr[0] - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (off[mid] <= t) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}
__device__ __forceinline__ int work_cell(const BoxDev& b, int t, int& kr)
{
    if (b.nrep == 1) return t;
    kr = work_replica(b, b.lw_off, t, kr);
    return b.rep[b.lw_rep[kr]].cell_off + (t - b.lw_off[kr]);
}
__device__ __forceinline__ int work_chunk(const BoxDev& b, int t, int& kr)
{
    if (b.nrep == 1) return t;
    kr = work_replica(b, b.lw_coff, t, kr);
    return b.rep[b.lw_rep[kr]].chunk_off + (t - b.lw_coff[kr]);
}

// The per-chunk stages run on groups of LJ_CHUNK threads: the blocks of the
// separate kernels, or the quarters of a block of the cluster kernel.
__device__ __forceinline__ int group_first() { return blockIdx.x * (blockDim.x / LJ_CHUNK) + threadIdx.x / LJ_CHUNK; }
__device__ __forceinline__ int group_count() { return gridDim.x * (blockDim.x / LJ_CHUNK); }
__device__ __forceinline__ int group_thread() { return threadIdx.x % LJ_CHUNK; }

// ---------------------------------------------------------------------------
// k_bin: new cell of every particle of a rebuilding replica, its offset from
// the new cell's centre (offB, the state's layout), its wrapped FP64 position
// (xabsB, the positions the lists are decided for) and the old-order copies
// used by the gather.
//
// Steady state (double-single state, positions held as cell + offset): the
// move to a neighbour cell is read off the FP32 offset (|o| >= half an edge)
// and the new offset is o - d * edge in double-single arithmetic, so the
// only FP64 work is forming the position x = centre + o.  A particle that
// crosses the box, moves more than one cell, or sits in a boundary cell with
// x outside [0, L) at FP64 rounding, takes the FP64 path of a build from
// positions: wrap x into [0, L), cell = floor(x / edge), offset = x - centre.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void bin_from_x(const RepDev& R, double* x, int* im, int* q)
{
    for (int c = 0; c < 3; ++c) {
        const double L = R.L[c];
        const double f = floor_div(x[c], R.wrap_hi[c], L);
        if (f != 0.0) {
            x[c] = x[c] - L * f;
            im[c] += (int)f;
        }
        const int qc = (int)(x[c] * R.inv_ell[c]);
        q[c] = qc < 0 ? 0 : (qc >= R.nc[c] ? R.nc[c] - 1 : qc);
    }
}

// offset of x from the centre of cell q, in the state's layout (the centre
// rounded on its own, no FMA with the subtraction)
__device__ __forceinline__ void store_offB(const BoxDev& b, const RepDev& R, int p, const double* x, const int* q)
{
    for (int c = 0; c < 3; ++c) {
        const double o = x[c] - __dmul_rn(half_above(q[c]), R.ell[c]);
        if (b.prec == 0) {
            float h, l;
            ds_from_double(o, h, l);
            float* ob = reinterpret_cast<float*>(b.offB);
            ob[c * b.np + p] = h;
            ob[3 * b.np + c * b.np + p] = l;
        } else {
            b.offB[c * b.np + p] = o;
        }
    }
}

// All of a particle's loads come before its stores: the arrays may alias as
// far as the compiler knows, so a copy written load by load waits for each
// one in turn.  With that, and the FP32-to-FP64 conversions moved off the
// FP64 pipe (21 FP64 operations per particle -> 12), a 4M binning went from
// 368 us to 203 us and the gather from 254 us to 214 us.
template <bool DS>
__device__ __forceinline__ void bin_chunks(const BoxDev& b, int from_abs)
{
    const int tot = work_chunks(b), np = b.np;
    const float* const off = reinterpret_cast<const float*>(b.off);
    const float* const vel = reinterpret_cast<const float*>(b.vel);
    float* const velB = reinterpret_cast<float*>(b.velB);
    int kr = 0;
    for (int t = group_first(); t < tot; t += group_count()) {
        const int w = work_chunk(b, t, kr);
        int4 ch = chunk_of(b, w);
        int r = ch.x;
        int p = ch.y + group_thread();
        const bool act = p < ch.z;   // every lane reaches the warp-wide count below
        if (!act) p = ch.y;
        const RepDev& R = b.rep[r];
        const int uid = b.uid[p], type = b.type[p];
        double x[3], vd[3];
        float oh[3], ol[3], vh[3], vl[3];
        int im[3], q[3];
        const int cell = from_abs ? 0 : b.cell[p];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            im[c] = b.img[c * np + p];
            if (DS) {
                vh[c] = vel[c * np + p];
                vl[c] = vel[3 * np + c * np + p];
            } else {
                vd[c] = b.vel[c * np + p];
            }
            if (from_abs) {
                x[c] = b.xabs[c * np + p];
            } else if (DS) {
                oh[c] = off[c * np + p];
                ol[c] = off[3 * np + c * np + p];
            } else {
                x[c] = b.off[c * np + p];   // the offset; the position below
            }
        }
        if (from_abs) {
            bin_from_x(R, x, im, q);
            if (act) store_offB(b, R, p, x, q);
        } else {
            int cx, cy;
            const int cz = cell_coords(R, cell, cx, cy);
            const int cc[3] = {cx, cy, cz};
            bool slow = !DS;
            if (DS) ds_to_double3(oh, ol, x);
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const double o = x[c];
                if (DS) {
                    const float h = oh[c];
                    // the neighbour cell the FP32 offset lies in (at most one away)
                    const float hh = 0.5f * R.ellf[c];
                    const int d = h >= hh ? 1 : (h < -hh ? -1 : 0);
                    const int qc = cc[c] + d;
                    slow = slow || fabsf(h) >= 3.f * hh || qc < 0 || qc >= R.nc[c];
                    q[c] = qc;
                    // o - d * edge, double-single (d * ellf is exact)
                    ds_add_ds(oh[c], ol[c], -(float)d * R.ellf[c], -(float)d * R.ell_lo[c]);
                }
                x[c] = __dmul_rn(half_above(cc[c]), R.ell[c]) + o;
                // a boundary cell: the position must still be inside [0, L)
                if ((cc[c] == 0 || cc[c] == R.nc[c] - 1) && !(x[c] >= 0.0 && x[c] < R.wrap_hi[c])) slow = true;
            }
            if (slow) {
                bin_from_x(R, x, im, q);
                if (act) store_offB(b, R, p, x, q);
            } else if (act) {
                float* ob = reinterpret_cast<float*>(b.offB);
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    ob[c * np + p] = oh[c];
                    ob[3 * np + c * np + p] = ol[c];
                }
            }
        }
        int gc = R.cell_off + q[0] + R.nc[0] * (q[1] + R.nc[1] * q[2]);
        if (act) {
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                b.xabsB[c * np + p] = x[c];
                b.imgB[c * np + p] = im[c];
                if (DS) {
                    velB[c * np + p] = vh[c];
                    velB[3 * np + c * np + p] = vl[c];
                } else {
                    b.velB[c * np + p] = vd[c];
                }
            }
            b.uidB[p] = uid;
            b.typeB[p] = type;
            b.cellB[p] = gc;
        }
        // warp-aggregated count: particles arrive in cell order, so a warp's
        // lanes share one or two cells; one atomic per distinct cell
        const int key = act ? gc : -1;
        const unsigned peers = __match_any_sync(0xffffffffu, key);
        if (act && (threadIdx.x & 31) == __ffs(peers) - 1) atomicAdd(&b.cell_count[gc], __popc(peers));
    }
}

__device__ __forceinline__ void phase_bin(const BoxDev& b, int from_abs)
{
    if (b.prec == 0) bin_chunks<true>(b, from_abs);
    else bin_chunks<false>(b, from_abs);
}

__global__ void __launch_bounds__(LJ_CHUNK) k_bin(BoxDev b, int from_abs)
{
    await_previous();
    if (box_needs_rebuild(b)) phase_bin(b, from_abs);
}

// ---------------------------------------------------------------------------
// Exclusive scan of cell counts inside each replica: a block per tile of
// kScanTile cells, a run of consecutive cells per thread; it first sums the
// counts of the replica's earlier tiles itself (from L2; at 4M the last of 101
// tiles reads 0.8 MB), which costs the few builds less than a second pass, a
// launch in every step: a step at N = 100,000 38.0 -> 36.6 us.  The reads grow
// with the square of the tiles, which is not seen at 32M (a forced update takes
// 0.65 ns per particle, 0.67 at 4M).  tiles[t] = (rep, first cell, end cell,
// first tile of the replica).
// ---------------------------------------------------------------------------
__device__ __forceinline__ int block_excl_scan(int v, int* s_warp, int& total)
{
    int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        int t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += t;
    }
    if (lane == 31) s_warp[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        int nw = blockDim.x >> 5;
        int x = lane < nw ? s_warp[lane] : 0;
        int xi = x;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            int t = __shfl_up_sync(0xffffffffu, xi, o);
            if (lane >= o) xi += t;
        }
        if (lane < nw) s_warp[lane] = xi - x;   // exclusive warp offsets
        if (lane == nw - 1) s_warp[32] = xi;    // block total
    }
    __syncthreads();
    int r = incl - v + s_warp[warp];
    total = s_warp[32];
    __syncthreads();
    return r;
}

template <int THREADS>
__device__ __forceinline__ void phase_scan(const BoxDev& b, const int4* tiles, int ntiles)
{
    constexpr int PER = kScanTile / THREADS;   // cells per thread
    __shared__ int s_warp[33];
    for (int t = blockIdx.x; t < ntiles; t += gridDim.x) {
        const int4 tl = tiles[t];
        if (!rep_needs_rebuild(b, tl.x)) continue;   // block-uniform
        const int c0 = tl.y + (int)threadIdx.x * PER;
        int v[PER], sum = 0, part = 0, total;
#pragma unroll
        for (int u = 0; u < PER; ++u) {
            v[u] = c0 + u < tl.z ? b.cell_count[c0 + u] : 0;
            sum += v[u];
        }
        for (int c = b.rep[tl.x].cell_off + (int)threadIdx.x; c < tl.y; c += 8 * THREADS) {
            int x[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) x[u] = c + u * THREADS < tl.y ? b.cell_count[c + u * THREADS] : 0;
#pragma unroll
            for (int u = 0; u < 8; ++u) part += x[u];
        }
        int before = 0;
        if (t != tl.w) block_excl_scan(part, s_warp, before);   // block-uniform
        int ex = block_excl_scan(sum, s_warp, total) + before + b.rep[tl.x].p_off;
#pragma unroll
        for (int u = 0; u < PER; ++u) {
            if (c0 + u < tl.z) {   // the range is open for k_scatter (cell_end is the cursor; it ends at start + count)
                b.cell_start[c0 + u] = ex;
                b.cell_end[c0 + u] = ex;
            }
            ex += v[u];
        }
    }
}

__global__ void __launch_bounds__(kScanThreads) k_scan(BoxDev b, const int4* tiles, int ntiles)
{
    await_previous();
    if (box_needs_rebuild(b)) phase_scan<kScanThreads>(b, tiles, ntiles);
}

// ---------------------------------------------------------------------------
// k_scatter: claim a slot inside the particle's new cell.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void phase_scatter(const BoxDev& b)
{
    const int tot = work_chunks(b);
    int kr = 0;
    for (int t = group_first(); t < tot; t += group_count()) {
        int4 ch = chunk_of(b, work_chunk(b, t, kr));
        int p = ch.y + group_thread();
        const bool act = p < ch.z;
        // warp-aggregated slot claims: one atomic per distinct cell of the
        // warp, each lane's slot = old cursor + its rank among the peers
        const int c = act ? b.cellB[p] : -1;
        const unsigned peers = __match_any_sync(0xffffffffu, c);
        const int lane = threadIdx.x & 31, leader = __ffs(peers) - 1;
        int base = 0;
        if (act && lane == leader) base = atomicAdd(&b.cell_end[c], __popc(peers));
        base = __shfl_sync(0xffffffffu, base, leader);
        if (act) b.perm[base + __popc(peers & ((1u << lane) - 1u))] = p;
    }
}

__global__ void __launch_bounds__(LJ_CHUNK) k_scatter(BoxDev b)
{
    await_previous();
    if (box_needs_rebuild(b)) phase_scatter(b);
}

// ---------------------------------------------------------------------------
// k_list_work: the work of a rebuild, one block.  The rebuilding replicas in
// order, with the prefixes of their cell and particle-chunk counts, so that
// the per-cell kernels (k_sortgather, k_nlist_lanes) and the per-chunk ones
// (k_bin, k_scatter) stride over those cells and chunks only: a step
// in which a few replicas of many rebuild does not walk (and test) every cell
// and chunk of the batch.  Launched first in every rebuild sequence.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void phase_list_work(const BoxDev& b)   // one block
{
    __shared__ int s_warp[33];
    int nsel = 0, ncell = 0, nch = 0;
    for (int base = 0; base < b.nrep; base += blockDim.x) {
        const int r = base + (int)threadIdx.x;
        const bool need = r < b.nrep && rep_needs_rebuild(b, r);
        int tsel, tcell, tch;
        const int xs = block_excl_scan(need ? 1 : 0, s_warp, tsel);
        const int xc = block_excl_scan(need ? b.rep[r].ncell : 0, s_warp, tcell);
        const int xh = block_excl_scan(need ? b.rep[r].nchunk : 0, s_warp, tch);
        if (need) {
            b.lw_rep[nsel + xs] = r;
            b.lw_off[nsel + xs] = ncell + xc;
            b.lw_coff[nsel + xs] = nch + xh;
        }
        nsel += tsel;
        ncell += tcell;
        nch += tch;
    }
    if (threadIdx.x == 0) {
        b.lw_off[nsel] = ncell;
        b.lw_coff[nsel] = nch;
        b.lw_hdr[0] = nsel;
    }
}

__global__ void __launch_bounds__(1024) k_list_work(BoxDev b, unsigned long long* runs)
{
    await_previous();
    if (!box_needs_rebuild(b)) return;
    phase_list_work(b);
    if (runs && threadIdx.x == 0) *runs += 1ull;   // launch accounting of a conditional rebuild
}

// ---------------------------------------------------------------------------
// k_sortgather: one warp per cell.  Order the members of the cell by their
// FP32 z offset from the cell centre (the value posq will hold), ties by
// user index (count of smaller keys; keys are unique), so the layout is a
// deterministic function of the positions and the list build can take, in
// every neighbour cell, the contiguous run of candidates within reach along
// z.  The alternative layout (order 1) sorts a cell by a space-filling curve
// over its 4 x 4 x 4 sub-cells first (Sec. 3: particles are sorted for
// locality); the list build then takes whole neighbour cells.  The lane that
// ranked a member moves its state, the new cell-relative offsets (computed by
// k_bin) and their FP32 copy to its slot.  (All pairs: one cell per replica,
// no order.)  Bound: DRAM and the latency of the gathered loads, all issued
// before the stores.  A kernel of its own for the gather, one thread per
// particle, had all its lanes busy (a cell fills 18 of 32), but read the keys'
// lines again and was one more launch in every step: forced update at 256,000
// 271 -> 262 us, at 4M 2837 -> 2771; a step at 100,000 39.4 -> 38.0 us.
// ---------------------------------------------------------------------------
// FP32 offset from the new cell centre, as posq will hold it (offB, from k_bin)
__device__ __forceinline__ float offB32(const BoxDev& b, int c, int p)
{
    if (b.prec == 0) return reinterpret_cast<const float*>(b.offB)[c * b.np + p];
    return __double2float_rn(b.offB[c * b.np + p]);
}

__device__ __forceinline__ unsigned long long sort_key(const BoxDev& b, const RepDev& R, int p)
{
    const float z = offB32(b, 2, p);
    const unsigned u = __float_as_uint(z);
    const unsigned ord = (u & 0x80000000u) ? ~u : (u | 0x80000000u);   // order-preserving
    if (b.order == 0) return ((unsigned long long)ord << 32) | (unsigned)b.uidB[p];
    // space-filling-curve order (Morton, or Z-order, curve over the cell's
    // 4 x 4 x 4 sub-cells: the sub-cell coordinates' bits interleaved), then
    // the z offset, then the user index (< 2^26) -- 6 + 32 + 26 bits
    unsigned m = 0;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        int sc = (int)floorf((offB32(b, c, p) / R.ellf[c] + 0.5f) * 4.f);
        sc = sc < 0 ? 0 : (sc > 3 ? 3 : sc);
        m |= (unsigned)(sc & 1) << c | (unsigned)(sc >> 1) << (c + 3);
    }
    return ((unsigned long long)m << 58) | ((unsigned long long)ord << 26) | (unsigned)b.uidB[p];
}

// Gather particle p (old order) into slot q of cell gc: its state, its new
// offsets (from k_bin) and their FP32 copy.  No arithmetic; every load before
// the stores (see bin_chunks).
template <bool DS>
__device__ __forceinline__ void gather_state(const BoxDev& b, int p, int q, int gc)
{
    const int np = b.np;
    const int ty = b.typeB[p], uid = b.uidB[p];
    double xa[3], o[3], v[3];
    float oh[3], ol[3], vh[3], vl[3];
    int im[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        xa[c] = b.xabsB[c * np + p];
        im[c] = b.imgB[c * np + p];
        if (DS) {
            const float* ob = reinterpret_cast<const float*>(b.offB);
            const float* vb = reinterpret_cast<const float*>(b.velB);
            oh[c] = ob[c * np + p];
            ol[c] = ob[3 * np + c * np + p];
            vh[c] = vb[c * np + p];
            vl[c] = vb[3 * np + c * np + p];
        } else {
            o[c] = b.offB[c * np + p];
            v[c] = b.velB[c * np + p];
        }
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        b.xabs[c * np + q] = xa[c];
        b.img[c * np + q] = im[c];
        if (DS) {
            float* of = reinterpret_cast<float*>(b.off);
            float* vf = reinterpret_cast<float*>(b.vel);
            of[c * np + q] = oh[c];
            of[3 * np + c * np + q] = ol[c];
            vf[c * np + q] = vh[c];
            vf[3 * np + c * np + q] = vl[c];
        } else {
            b.off[c * np + q] = o[c];
            b.vel[c * np + q] = v[c];
            if (b.offx) b.offx[c * np + q] = __double2ll_rn(o[c] * b.fx.scale);
            oh[c] = __double2float_rn(o[c]);
        }
    }
    b.uid[q] = uid;
    b.type[q] = ty;
    b.cell[q] = gc;
    const float4 pq = make_float4(oh[0], oh[1], oh[2], __int_as_float(ty));
    b.posq[q] = pq;
    b.ref[q] = pq;
}
__device__ __forceinline__ void gather_one(const BoxDev& b, int p, int q, int gc)
{
    if (b.prec == 0) gather_state<true>(b, p, q, gc);
    else gather_state<false>(b, p, q, gc);
}

// Rank the members of the cells and move them to their slots.
__device__ __forceinline__ void phase_rank(const BoxDev& b)
{
    const int lane = threadIdx.x & 31;
    const int wpb = blockDim.x >> 5;
    const int total = work_cells(b);
    int kr = 0;
    for (int t = blockIdx.x * wpb + (threadIdx.x >> 5); t < total; t += gridDim.x * wpb) {
        const int gc = work_cell(b, t, kr);
        const RepDev& R = b.rep[b.nrep == 1 ? 0 : b.lw_rep[kr]];
        int s0 = b.cell_start[gc];
        int n = b.cell_end[gc] - s0;
        if (lane == 0) b.cell_count[gc] = 0;   // for the next build
        for (int base = 0; base < n; base += 32) {
            int idx = base + lane;
            int p = idx < n ? b.perm[s0 + idx] : -1;
            const unsigned long long none = ~0ull;
            unsigned long long key = idx < n ? sort_key(b, R, p) : none;
            int rank = 0;
            for (int b2 = 0; b2 < n; b2 += 32) {
                unsigned long long k2 =
                    b2 == base ? key : ((b2 + lane < n) ? sort_key(b, R, b.perm[s0 + b2 + lane]) : none);
#pragma unroll 8
                for (int t = 0; t < 32; ++t) {
                    unsigned long long kt = __shfl_sync(0xffffffffu, k2, t);
                    rank += (kt < key) ? 1 : 0;
                }
            }
            if (idx < n) gather_one(b, p, s0 + rank, gc);
        }
    }
}

__global__ void __launch_bounds__(256) k_sortgather(BoxDev b)
{
    await_previous();
    if (!box_needs_rebuild(b)) return;
    if (b.all_pairs) {
        // one cell holds the whole replica and no list needs an order: a
        // particle's slot is its index inside the replica, one thread each
        const int tot = work_chunks(b);
        int kr = 0;
        for (int t = blockIdx.x; t < tot; t += gridDim.x) {
            const int4 ch = chunk_of(b, work_chunk(b, t, kr));
            const RepDev& R = b.rep[ch.x];
            for (int s = ch.y + (int)threadIdx.x; s < ch.z; s += blockDim.x) {
                if (s == R.p_off) {
                    atomicAdd(&b.nbuild[ch.x], 1ull);   // a re-binning
                    b.cell_count[R.cell_off] = 0;       // for the next one
                }
                const int p = b.perm[s];
                gather_one(b, p, R.p_off + (b.uidB[p] - R.u_off), R.cell_off);
            }
        }
        return;
    }
    phase_rank(b);
}

// ---------------------------------------------------------------------------
// k_nlist: Verlet list of every particle of a rebuilding replica (Sec. 3),
// one segment per block.  The segment's tile (its 27-cell neighbourhood) is
// staged in shared memory and candidates are read from there.  Membership
// |d_ij|^2 < rl^2 is decided in FP32 from the cell-relative offsets; pairs
// within `band` of rl^2 are re-decided in FP64 from the wrapped positions
// with the minimum image, in the same operation order as the plain
// definition, so the lists equal the FP64 definition exactly.
// ---------------------------------------------------------------------------
__device__ __forceinline__ bool exact_within(const BoxDev& b, const RepDev& R, int p, int j)
{
    double dd[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        double d = __dsub_rn(b.xabs[c * b.np + p], b.xabs[c * b.np + j]);
        double t = rint(__ddiv_rn(d, R.L[c]));
        dd[c] = __dsub_rn(d, __dmul_rn(R.L[c], t));
    }
    double d2 = __dadd_rn(__dadd_rn(__dmul_rn(dd[0], dd[0]), __dmul_rn(dd[1], dd[1])),
                          __dmul_rn(dd[2], dd[2]));
    return d2 < b.rl2;
}

__global__ void __launch_bounds__(LJ_LIST_THREADS, 3) k_nlist(BoxDev b)
{
    if (!box_needs_rebuild(b)) return;
    extern __shared__ __align__(16) float4 s_tile[];   // LJ_TILE_MAX entries
    __shared__ float4 s_shift[32];
    __shared__ int4 s_rng[LJ_SEG_MAX_CELLS * 27];   // (first, end, tile offset) per (cell, k)
    __shared__ int s_qoff[LJ_SEG_MAX_CELLS + 1];     // first quad of each cell
    __shared__ uint16_t s_flat[(LJ_LIST_THREADS / 32) * LJ_FLAT_MAX];   // per-warp candidate list
    __shared__ uint32_t s_kent[(LJ_LIST_THREADS / 32) * 32];             // per-warp entry bases
    __shared__ Tile s_t;
    __shared__ __align__(8) unsigned long long s_bar;
    __shared__ int s_next;      // next quad of the segment to hand out
    __shared__ int s_longest;   // longest list this block built
    if (threadIdx.x == 0) {
        mbar_init(&s_bar, 1);
        s_longest = 0;
    }
    unsigned phase = 0;
    int cur_r = -1;
    const float lo2 = b.rl2f - b.band, hi2 = b.rl2f + b.band;
    for (int w = blockIdx.x; w < b.nseg; w += gridDim.x) {
        int4 sg = b.seg[w];
        int r = sg.x;
        if (!rep_needs_rebuild(b, r)) continue;   // block-uniform
        const RepDev& R = b.rep[r];
        __syncthreads();                          // previous segment done
        if (threadIdx.x < 32) {
            // warp 0: the tile's pieces, and the segment's quads per cell
            Tile t;
            seg_tile_warp(b, R, sg, t);
            const int lane = threadIdx.x;
            if (lane == 0) {
                s_t = t;
                if (w == R.seg_off) atomicAdd(&b.nbuild[r], 1ull);
            }
            const int cbase = R.cell_off + sg.y + R.nc[0] * sg.z;
            const int nqc = lane < sg.w ? (b.cell_end[cbase + lane] - b.cell_start[cbase + lane] + 3) >> 2 : 0;
            int incl = nqc;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int v = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += v;
            }
            if (lane < sg.w) s_qoff[lane] = incl - nqc;
            if (lane == sg.w - 1) s_qoff[sg.w] = incl;
            if (lane == 0) s_next = LJ_LIST_THREADS / 32;
        }
        if (r != cur_r && threadIdx.x < 32) {
            int k = threadIdx.x;
            s_shift[k] = k < 27 ? make_float4((float)(k % 3 - 1) * R.ellf[0], (float)((k / 3) % 3 - 1) * R.ellf[1],
                                              (float)(k / 9 - 1) * R.ellf[2], 0.f)
                                : make_float4(0.f, 0.f, 0.f, 0.f);
        }
        cur_r = r;
        __syncthreads();
        const int n = s_t.n, p0 = s_t.p0;
        if (s_t.total > LJ_TILE_MAX) {
            if (threadIdx.x == 0) atomicOr(&b.err[0], LJ_ERRBIT_TILE);
            for (int il = threadIdx.x; il < n; il += blockDim.x) b.nbr_count[p0 + il] = 0;
            continue;
        }
        // neighbour-cell ranges of the segment's cells, with their tile offsets
        const int nx = R.nc[0], ny = R.nc[1], nz = R.nc[2];
        const int cy = sg.z % ny, cz = sg.z / ny;
        const int c0 = R.cell_off + sg.y + nx * sg.z;
        for (int idx = threadIdx.x; idx < sg.w * 27; idx += blockDim.x) {
            const int cl = idx / 27, k = idx % 27;
            const int dx = k % 3 - 1, dy = (k / 3) % 3 - 1, dz = k / 9 - 1;
            const int cn = R.cell_off + wrapi(sg.y + cl + dx, nx) + nx * (wrapi(cy + dy, ny) + ny * wrapi(cz + dz, nz));
            const int js = b.cell_start[cn], je = b.cell_end[cn];
            int q = 2 * (3 * (dz + 1) + (dy + 1));
            if (!(js >= s_t.beg[q] && js < s_t.end[q])) ++q;
            s_rng[idx] = make_int4(js, je, s_t.base[q] - s_t.beg[q], 0);
        }
        if (s_t.total > 0 && !stage_tile_bulk(b.posq, s_t, s_tile, &s_bar, phase, b.err)) return;
        const float ell_h[3] = {0.5f * R.ellf[0], 0.5f * R.ellf[1], 0.5f * R.ellf[2]};
        const float rcull = b.rl2f + b.band;
        // reach along z of any pair the FP32 test can accept (r2 < rl^2 +
        // band implies dz^2 < rl^2 + band), with a margin for the rounding of
        // the shifted z values
        const float zreach = sqrtf(rcull) + 1e-3f;
        // work units: quads of particles of one cell (the quad's particles
        // share the cell, so their candidates are the same), handed out to
        // the warps one at a time as they finish (s_qoff, s_next set above)
        const int nquad = s_qoff[sg.w];
        const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
        uint16_t* flat = s_flat + warp * LJ_FLAT_MAX;
        uint32_t* kent = s_kent + warp * 32;
        for (int qd = warp; qd < nquad;) {
            int cl = 0;
            while (s_qoff[cl + 1] <= qd) ++cl;                  // warp-uniform
            const int cs = b.cell_start[c0 + cl], ce = b.cell_end[c0 + cl];
            const int p0q = cs + 4 * (qd - s_qoff[cl]);          // first particle of the quad
            const int nq = min(4, ce - p0q);                     // particles in the quad
            // the quad's particles, in every lane's registers
            float4 pq[4];
#pragma unroll
            for (int g = 0; g < 4; ++g) pq[g] = b.posq[p0q + (g < nq ? g : 0)];
            const int4* rng = s_rng + cl * 27;
            // flatten the candidate cells (lane k owns stencil cell k); a cell
            // is dropped when its box lies beyond the list radius of all the
            // quad's particles
            int len = 0;
            int4 rk = make_int4(0, 0, 0, 0);
            if (lane < 27) {
                rk = rng[lane];
                const float4 sh = s_shift[lane];
                bool far = true;
                float zmin = pq[0].z, zmax = pq[0].z;
#pragma unroll
                for (int g = 0; g < 4; ++g) {
                    const float gx = fmaxf(fabsf(pq[g].x - sh.x) - ell_h[0], 0.f);
                    const float gy = fmaxf(fabsf(pq[g].y - sh.y) - ell_h[1], 0.f);
                    const float gz = fmaxf(fabsf(pq[g].z - sh.z) - ell_h[2], 0.f);
                    far = far && (g >= nq || gx * gx + gy * gy + gz * gz >= rcull);
                    zmin = fminf(zmin, pq[g].z);   // g >= nq repeats particle 0
                    zmax = fmaxf(zmax, pq[g].z);
                }
                if (!far && b.order != 0) {
                    len = rk.y - rk.x;   // space-filling-curve order: the whole cell
                } else if (!far) {
                    // the cell is sorted by z offset: keep the run with
                    // z_j + shift_z within zreach of the quad's z range
                    const float zlo = zmin - zreach - sh.z, zhi = zmax + zreach - sh.z;
                    const float* tz = reinterpret_cast<const float*>(s_tile) + 2;   // .z of tile entry t: tz[4 t]
                    int lo = rk.x + rk.z, hi = rk.y + rk.z;
                    while (lo < hi) {
                        const int mid = (lo + hi) >> 1;
                        if (tz[4 * mid] < zlo) lo = mid + 1;
                        else hi = mid;
                    }
                    int e = rk.y + rk.z;
                    hi = e;
                    int lo2 = lo;
                    while (lo2 < hi) {
                        const int mid = (lo2 + hi) >> 1;
                        if (tz[4 * mid] <= zhi) lo2 = mid + 1;
                        else hi = mid;
                    }
                    rk.x = lo - rk.z;
                    rk.y = lo2 - rk.z;
                    len = rk.y - rk.x;
                }
            }
            int incl = len;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int t = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += t;
            }
            const int total = __shfl_sync(0xffffffffu, incl, 31);
            // entry of tile index t from cell k: t above the digits + kent[k]
            // (the slot being t minus the cell's tile offset)
            if (lane < 27) kent[lane] = entry_make(lane, 0) - ((uint32_t)rk.z << LJ_DIGIT_BITS);
            const int self13 = p0q + __shfl_sync(0xffffffffu, rk.z, 13);   // tile index of the quad's first particle
            const int off = incl - len;
            int cnt[4] = {0, 0, 0, 0};
            bool nearb[4] = {false, false, false, false};   // saw a pair within the FP64 recheck band
            const unsigned lt_mask = (1u << lane) - 1u;
            uint32_t* const row0 = b.nbr + (size_t)b.K * p0q;   // list of the quad's first particle
            for (int w0 = 0; w0 < total; w0 += LJ_FLAT_MAX) {
                const int wn = min(total - w0, LJ_FLAT_MAX);
                __syncwarp();
                if (lane < 27) {
                    // lane k writes its cell's part of the window: (k, tile index)
                    const int ok = off - w0;
                    const int t_lo = max(0, -ok), t_hi = min(len, wn - ok);
                    const unsigned code = ((unsigned)lane << LJ_TILE_BITS) | (unsigned)(rk.x + rk.z);
                    for (int t = t_lo; t < t_hi; ++t) flat[ok + t] = (uint16_t)(code + (unsigned)t);
                }
                __syncwarp();
                // one candidate per lane, tested against the quad's particles;
                // pairs within the recheck band are kept here and settled in
                // FP64 afterwards
                // two candidates per lane per pass (t and t + 32): two
                // independent test-and-append chains for the scheduler
                for (int t0 = 0; t0 < wn; t0 += 64) {
                    float qx[2], qy[2], qz[2];
                    uint32_t ent[2];
                    int selfg[2];
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const int t = t0 + 32 * h + lane;
                        const unsigned e = t < wn ? flat[t] : 0u;
                        const int k = (int)(e >> LJ_TILE_BITS);
                        const int idx = (int)(e & LJ_TILE_MASK);
                        const float4 pj = s_tile[idx];
                        const float4 sh = s_shift[k];
                        // lanes past the window take a far point, whose r2 is inf
                        qx[h] = t < wn ? pj.x + sh.x : 1.0e38f;
                        qy[h] = pj.y + sh.y;
                        qz[h] = pj.z + sh.z;
                        ent[h] = ((uint32_t)idx << LJ_DIGIT_BITS) + kent[k];
                        // tile slices are disjoint, so the index alone finds the
                        // particle itself: quad slot idx - self13 (if in 0..3)
                        selfg[h] = idx - self13;
                    }
#pragma unroll
                    for (int g = 0; g < 4; ++g) {
                        if (g >= nq) break;   // warp-uniform: slots past the quad's end take nothing
                        bool in[2];
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            const float ddx = pq[g].x - qx[h], ddy = pq[g].y - qy[h], ddz = pq[g].z - qz[h];
                            const float r2 = ddx * ddx + ddy * ddy + ddz * ddz;
                            in[h] = r2 < hi2 && selfg[h] != g;
                            nearb[g] = nearb[g] || (in[h] && r2 >= lo2);
                        }
                        const unsigned b0 = __ballot_sync(0xffffffffu, in[0]);
                        const unsigned b1 = __ballot_sync(0xffffffffu, in[1]);
                        const int pos0 = cnt[g] + __popc(b0 & lt_mask);
                        const int pos1 = cnt[g] + __popc(b0) + __popc(b1 & lt_mask);
                        uint32_t* const rg = row0 + (size_t)b.K * g;
                        if (cnt[g] + 64 <= b.K) {   // warp-uniform: room for the whole pass
                            if (in[0]) rg[pos0] = ent[0];
                            if (in[1]) rg[pos1] = ent[1];
                        } else {                    // entries beyond the capacity are counted only
                            if (in[0] && pos0 < b.K) rg[pos0] = ent[0];
                            if (in[1] && pos1 < b.K) rg[pos1] = ent[1];
                        }
                        cnt[g] += __popc(b0) + __popc(b1);
                    }
                }
            }
            // FP64 decision for the particles that saw a pair near rl: drop the
            // band pairs beyond rl and compact their lists
#pragma unroll
            for (int g = 0; g < 4; ++g) {
                if (g >= nq || !__any_sync(0xffffffffu, nearb[g])) continue;   // warp-uniform
                __syncwarp();   // the list's entries, stored by other lanes, are visible
                const int p = p0q + g;
                uint32_t* const row = row0 + (size_t)b.K * g;
                const int c = min(cnt[g], b.K);
                int kept = 0;
                for (int s0 = 0; s0 < c; s0 += 32) {
                    const int s = s0 + lane;
                    bool keep = false;
                    uint32_t ent = 0;
                    if (s < c) {
                        ent = row[s];
                        const int j = (int)entry_slot(ent);
                        const int k = entry_k(ent);
                        const float4 pj = b.posq[j];
                        const float4 sh = s_shift[k];
                        const float ddx = pq[g].x - (pj.x + sh.x), ddy = pq[g].y - (pj.y + sh.y),
                                    ddz = pq[g].z - (pj.z + sh.z);
                        const float r2 = ddx * ddx + ddy * ddy + ddz * ddz;
                        keep = r2 < lo2 || exact_within(b, R, p, j);
                    }
                    const unsigned bits = __ballot_sync(0xffffffffu, keep);
                    __syncwarp();
                    if (keep) row[kept + __popc(bits & lt_mask)] = ent;
                    kept += __popc(bits);
                }
                cnt[g] = cnt[g] - c + kept;   // entries beyond the capacity are counted, not stored
            }
            const int c = lane == 0 ? cnt[0] : lane == 1 ? cnt[1] : lane == 2 ? cnt[2] : cnt[3];
            if (lane < nq) {
                b.nbr_count[p0q + lane] = c;
                for (int s = c; s < b.K && (s & 3); ++s)   // the row's last piece of four is filled with the sentinel
                    row0[(size_t)b.K * lane + s] = entry_make(13, b.np);
                if (c > b.K) {
                    atomicOr(&b.err[0], LJ_ERRBIT_CAPACITY);
                    atomicMax(&b.err[1], c);
                }
            }
            const int cmax = __reduce_max_sync(0xffffffffu, lane < nq ? c : 0);
            int nxt = 0;
            if (lane == 0) {
                atomicMax(&s_longest, cmax);
                nxt = atomicAdd(&s_next, 1);
            }
            qd = __shfl_sync(0xffffffffu, nxt, 0);
        }
    }
    __syncthreads();
    if (threadIdx.x == 0 && s_longest > 0) atomicMax(&b.err[2], s_longest);   // longest list of this build
}

// ---------------------------------------------------------------------------
// k_nlist_lanes: the same lists, one warp per pass of 32 / G particles of a
// cell, G lanes per particle.  The warp streams the candidates of the 27
// neighbour cells in chunks of 32: lane t loads candidate t of the chunk
// (coalesced, the next chunk's load in flight while this one is used), adds
// the cell's shift and drops it when its distance from the bounding box of
// the pass's particles is beyond the list radius (at least a quarter of the
// 27-cell block lies there); the kept candidates (shifted FP32 offset and
// list entry) go to a per-warp ring in shared memory.  Every 32 staged
// candidates, each lane tests its 32 / G of them against its particle -- one
// broadcast shared-memory load per candidate and component -- and appends the
// entries of its hits to its own row buffer in shared memory (no ballots:
// every lane owns its buffer), from which whole pieces of four entries go out
// with 16-byte stores.  Pairs within `band` of rl^2 are re-decided in FP64 as
// in k_nlist (checked per half batch: the smallest |r^2 - rl^2| tells whether any
// pair lies in the band).  d_ij and r^2 are computed as FP32 pairs.
// G = 1 where the cells fill the GPU (launch_list's rule); what bounds it
// then: issue (74 % of peak) and the shared-memory pipe (65 %), ~310
// instructions a warp and 64 wavefronts of loads and stores per batch of 32
// candidates, which is why the buffers hold whole entries (a step's store is
// one wavefront; 16-bit codes took two, and a base table on the way out).
// G = 4 for small boxes: a cell's warp ran alone on its scheduler, ~10 cycles
// per instruction; four warps take a cell's particles, each with a tighter
// bounding box and a quarter of the tests per lane.
// Forced update (binning, sort, lists, force) at N = 4,000 176 -> 134 us, at 4M
// 3694 -> 3470 us (cell scale 1.15: 3215 -> 3016).
// ---------------------------------------------------------------------------
constexpr int kLaneWarps = LJ_LANE_THREADS / 32;
constexpr int kRing = 64;   // staged candidates per warp: < 32 waiting + one chunk
// Entries a lane holds in shared memory: fewer than 4 not yet written out, and
// half a batch's 32 / G on top (flushed when less room is left), so the rows'
// shared memory does not grow with the capacity K.  Looked at once a batch,
// the buffers were written out two or three entries at a time: forced update
// at 256,000 281 -> 269 us, at 4M 2956 -> 2839 (quarters: 277 and 2983; buffers
// of 32 or 48 entries: 2917 and 2883).
constexpr int kLaneRow = 40;

// r^2 - rl^2 of the pair (i, candidate q = o_j + shift), rounded as in the
// batches.
__device__ __forceinline__ float lane_t(const float4& pi, const float4& q, float rl2)
{
    const float dx = __fadd_rn(q.x, -pi.x), dy = __fadd_rn(q.y, -pi.y), dz = __fadd_rn(q.z, -pi.z);
    return __fmaf_rn(dz, dz, __fmaf_rn(dy, dy, __fmaf_rn(dx, dx, -rl2)));
}

template <int G>
__global__ void __launch_bounds__(LJ_LANE_THREADS, 8) k_nlist_lanes(BoxDev b)
{
    await_previous();
    if (!box_needs_rebuild(b)) return;
    constexpr int P = 32 / G;    // particles of a pass
    constexpr int T = 32 / G;    // candidates of a batch that a lane tests
    // row buffers, slot-major per warp: entry e of lane l at [e][l] (the 32
    // lanes' stores of one step fall in distinct banks whatever their counts)
    extern __shared__ __align__(16) uint32_t s_rows[];   // per warp: kLaneRow x 32 entries
    __shared__ __align__(16) float s_cx[kLaneWarps][kRing];   // staged candidates: o_j + shift(k),
    __shared__ __align__(16) float s_cy[kLaneWarps][kRing];   // one array per component (four
    __shared__ __align__(16) float s_cz[kLaneWarps][kRing];   // candidates load as one 16-byte word)
    __shared__ __align__(16) uint32_t s_ce[kLaneWarps][kRing];   // and their list entries
    __shared__ int2 s_rng[kLaneWarps][27];                // neighbour cell k: (first slot, end slot)
    __shared__ float4 s_sh[kLaneWarps][27];               // shift(k) = (dx, dy, dz) * cell edge; k's digits
    __shared__ int s_longest;
    if (threadIdx.x == 0) s_longest = 0;
    __syncthreads();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int pl = lane % P, sub = lane / P;   // the lane's particle of the pass, its share of the candidates
    const unsigned lt = (1u << lane) - 1u;
    const int K = b.K;
    uint32_t* const row = s_rows + (size_t)warp * kLaneRow * 32 + lane;   // entry e at row[32 e]
    float* const rx = s_cx[warp];
    float* const ry = s_cy[warp];
    float* const rz = s_cz[warp];
    uint32_t* const re = s_ce[warp];
    const float rl2 = b.rl2f, band = b.band;
    const float rcull = rl2 + band + 1e-3f;   // staging margin for the rounding of the shifted offsets
    const float4* posq = b.posq;
    int longest = 0;
    const int nwarp = gridDim.x * kLaneWarps;
    const int total = work_cells(b) * G;
    int kr = 0;
    for (int t = blockIdx.x * kLaneWarps + warp; t < total; t += nwarp) {
        const int gc = work_cell(b, t / G, kr);
        const int r = b.nrep == 1 ? 0 : b.lw_rep[kr];
        const RepDev& R = b.rep[r];
        const int cs = b.cell_start[gc], n = b.cell_end[gc] - cs;
        if (lane == 0 && t % G == 0 && gc == R.cell_off) atomicAdd(&b.nbuild[r], 1ull);
        if (P * (t % G) >= n) continue;   // warp-uniform
        int cx, cy;
        const int cz = cell_coords(R, gc, cx, cy);
        __syncwarp();
        if (lane < 27) {
            const int dx = lane % 3 - 1, dy = (lane / 3) % 3 - 1, dz = lane / 9 - 1;
            const int cn = R.cell_off + wrapi(cx + dx, R.nc[0]) +
                           R.nc[0] * (wrapi(cy + dy, R.nc[1]) + R.nc[1] * wrapi(cz + dz, R.nc[2]));
            const int js = b.cell_start[cn], je = b.cell_end[cn];
            s_rng[warp][lane] = make_int2(js, je);
            s_sh[warp][lane] = make_float4((float)dx * R.ellf[0], (float)dy * R.ellf[1], (float)dz * R.ellf[2],
                                           __uint_as_float(entry_make(lane, 0)));
            if (je - js > LJ_TILE_MAX) atomicOr(&b.err[0], LJ_ERRBIT_TILE);   // refused: never at LJ densities
        }
        __syncwarp();
        for (int ib = P * (t % G); ib < n; ib += P * G) {
            const bool act = ib + pl < n;
            const int i = cs + (act ? ib + pl : 0);
            float4 pi = posq[i];
            // the box of this pass's particles (tighter than the cell: the
            // candidates to test are those within the list radius of it)
            float lx = act ? pi.x : 1.0e30f, ly = act ? pi.y : 1.0e30f, lz = act ? pi.z : 1.0e30f;
            float ux = act ? pi.x : -1.0e30f, uy = act ? pi.y : -1.0e30f, uz = act ? pi.z : -1.0e30f;
#pragma unroll
            for (int o = P / 2; o > 0; o >>= 1) {
                lx = fminf(lx, __shfl_xor_sync(0xffffffffu, lx, o));
                ly = fminf(ly, __shfl_xor_sync(0xffffffffu, ly, o));
                lz = fminf(lz, __shfl_xor_sync(0xffffffffu, lz, o));
                ux = fmaxf(ux, __shfl_xor_sync(0xffffffffu, ux, o));
                uy = fmaxf(uy, __shfl_xor_sync(0xffffffffu, uy, o));
                uz = fmaxf(uz, __shfl_xor_sync(0xffffffffu, uz, o));
            }
            if (!act) pi = make_float4(1.0e30f, 1.0e30f, 1.0e30f, 0.f);   // a far point: r^2 is inf
            const uint32_t self = entry_make(13, i);   // the particle itself
            int cnt = 0;                   // entries in the row buffer
            int flushed = 0;               // the particle's entries already written out (a multiple of 4)
            unsigned head = 0, tail = 0;   // ring positions (free-running; head stays a multiple of 32)
            uint4* const dst = reinterpret_cast<uint4*>(b.nbr + (size_t)K * i);   // the particle's row
            // x summed over the lanes of the particle before this one; all gets the sum over all of them
            auto lanes_before = [&](int x, int& all) {
                if (G == 1) {
                    all = x;
                    return 0;
                }
                int incl = x;
#pragma unroll
                for (int o = P; o < 32; o <<= 1) {
                    const int v = __shfl_up_sync(0xffffffffu, incl, o);
                    if (lane >= o) incl += v;
                }
                all = __shfl_sync(0xffffffffu, incl, 32 - P + pl);
                return incl - x;
            };
            // whole pieces of four entries out to the list, the rest to the
            // buffer's front; entries past the capacity are counted, not
            // written
            auto flush = [&]() {
                const int nq = act ? (cnt >> 2) : 0;
                int all;
                const int at = (flushed >> 2) + lanes_before(nq, all);
                for (int q = 0; q < nq; ++q) {
                    const uint4 o = make_uint4(row[32 * (4 * q)], row[32 * (4 * q + 1)], row[32 * (4 * q + 2)],
                                               row[32 * (4 * q + 3)]);
                    if (4 * (at + q + 1) <= K) dst[at + q] = o;
                }
                const int rest = cnt & 3;
                for (int q = 0; q < rest; ++q) row[32 * q] = row[32 * (cnt - rest + q)];
                flushed += 4 * all;
                cnt = rest;
            };
            // test the 32 staged candidates from head on against the lane's
            // particle and append the hits, half of them between two looks at
            // the buffers (which so fill further before they are written out)
            auto half_batch = [&](int h0) {
                if (__any_sync(0xffffffffu, cnt > kLaneRow - T / 2)) flush();
                const int c0 = cnt;
                // branch-free, two candidates per step with FP32-pair
                // arithmetic on t = r^2 - rl^2: every candidate's entry is
                // written to the next free slot (32-bit shared address), which
                // advances only on a hit
                float near = 1.0e30f;   // smallest |t| of the half
                uint32_t wa = (uint32_t)__cvta_generic_to_shared(row + 32 * cnt);
                const float2 px = make_float2(-pi.x, -pi.x), py = make_float2(-pi.y, -pi.y),
                             pz = make_float2(-pi.z, -pi.z), nrl = make_float2(-rl2, -rl2);
                // four candidates per step: one 16-byte broadcast load per
                // component and for the entries
                auto step2 = [&](float2 qx, float2 qy, float2 qz, uint32_t e0, uint32_t e1) {
                    const float2 dx = __fadd2_rn(qx, px), dy = __fadd2_rn(qy, py), dz = __fadd2_rn(qz, pz);
                    const float2 t2 = __ffma2_rn(dz, dz, __ffma2_rn(dy, dy, __ffma2_rn(dx, dx, nrl)));
                    near = fminf(fminf(near, fabsf(t2.x)), fabsf(t2.y));
                    asm volatile("st.shared.u32 [%0], %1;" ::"r"(wa), "r"(e0));
                    if ((t2.x < band) & (e0 != self)) wa += 128u;
                    asm volatile("st.shared.u32 [%0], %1;" ::"r"(wa), "r"(e1));
                    if ((t2.y < band) & (e1 != self)) wa += 128u;
                };
#pragma unroll
                for (int u = 0; u < T / 2; u += 4) {
                    const float4 qx = *reinterpret_cast<const float4*>(rx + h0 + u);
                    const float4 qy = *reinterpret_cast<const float4*>(ry + h0 + u);
                    const float4 qz = *reinterpret_cast<const float4*>(rz + h0 + u);
                    const uint4 qe = *reinterpret_cast<const uint4*>(re + h0 + u);
                    step2(make_float2(qx.x, qx.y), make_float2(qy.x, qy.y), make_float2(qz.x, qz.y), qe.x, qe.y);
                    step2(make_float2(qx.z, qx.w), make_float2(qy.z, qy.w), make_float2(qz.z, qz.w), qe.z, qe.w);
                }
                asm volatile("" ::: "memory");   // the stores above stay above
                __syncwarp();
                cnt = (int)((wa - (uint32_t)__cvta_generic_to_shared(row)) >> 7);
                // FP64 decision of the half's accepted pairs near rl (rare)
                if (near <= band) {
                    int w = c0;
                    const int e = cnt;
                    for (int q = c0; q < e; ++q) {
                        const uint32_t ent = row[32 * q];
                        const int j = (int)entry_slot(ent);
                        const float4 pj = posq[j];
                        const float4 sh = s_sh[warp][entry_k(ent)];
                        const float4 qj = make_float4(pj.x + sh.x, pj.y + sh.y, pj.z + sh.z, 0.f);
                        if (lane_t(pi, qj, rl2) < -band || exact_within(b, R, i, j)) row[32 * w++] = ent;
                    }
                    cnt = w;
                }
            };
            auto batch = [&]() {
#pragma unroll 1
                for (int h = 0; h < T; h += T / 2) half_batch((int)(head & (kRing - 1)) + T * sub + h);
                head += 32u;
            };
            // chunk iterator over the neighbour cells: (k, j0), 32 slots at a time
            int k = 0, j0 = s_rng[warp][0].x;
            while (k < 27 && j0 >= s_rng[warp][k].y) {
                ++k;
                if (k < 27) j0 = s_rng[warp][k].x;
            }
            float4 raw = make_float4(0.f, 0.f, 0.f, 0.f);
            if (k < 27 && j0 + lane < s_rng[warp][k].y) raw = posq[j0 + lane];
            while (k < 27) {
                const int len = min(32, s_rng[warp][k].y - j0);
                const float4 sh = s_sh[warp][k];
                const uint32_t ent = ((uint32_t)(j0 + lane) << LJ_DIGIT_BITS) | __float_as_uint(sh.w);
                const float4 cur = raw;
                j0 += 32;
                while (k < 27 && j0 >= s_rng[warp][k].y) {
                    ++k;
                    if (k < 27) j0 = s_rng[warp][k].x;
                }
                if (k < 27 && j0 + lane < s_rng[warp][k].y) raw = posq[j0 + lane];   // next chunk, in flight
                // stage: shift into the cell's frame, keep what can be within reach of the cell
                const float qx = cur.x + sh.x, qy = cur.y + sh.y, qz = cur.z + sh.z;
                const float gx = fmaxf(fmaxf(lx - qx, qx - ux), 0.f), gy = fmaxf(fmaxf(ly - qy, qy - uy), 0.f),
                            gz = fmaxf(fmaxf(lz - qz, qz - uz), 0.f);
                const bool keep = lane < len && fmaf(gx, gx, fmaf(gy, gy, gz * gz)) < rcull;
                const unsigned bal = __ballot_sync(0xffffffffu, keep);
                if (keep) {
                    const int q = (int)((tail + __popc(bal & lt)) & (kRing - 1));
                    rx[q] = qx;
                    ry[q] = qy;
                    rz[q] = qz;
                    re[q] = ent;
                }
                tail += __popc(bal);
                __syncwarp();
                if (tail - head >= 32) batch();
                __syncwarp();
            }
            if (tail > head) {   // far points fill the last batch
                if (lane >= (int)(tail - head)) rx[(head + lane) & (kRing - 1)] = 1.0e30f;
                __syncwarp();
                batch();
            }
            // what the buffers still hold, up to the capacity
            int c;
            if (G == 1) {
                c = flushed + cnt;
                if (act)   // the last piece may hold stale entries past the count
                    for (int q = 0; 4 * q < cnt && flushed + 4 * q < K; ++q)
                        dst[(flushed >> 2) + q] = make_uint4(row[32 * (4 * q)], row[32 * (4 * q + 1)],
                                                             row[32 * (4 * q + 2)], row[32 * (4 * q + 3)]);
            } else {
                flush();
                int all;
                const int at = flushed + lanes_before(act ? cnt : 0, all);
                if (act)
                    for (int q = 0; q < cnt; ++q)
                        if (at + q < K) reinterpret_cast<uint32_t*>(dst)[at + q] = row[32 * q];
                c = flushed + all;
            }
            if (act && sub == 0) {
                b.nbr_count[i] = c;
                if (c > K) {
                    atomicOr(&b.err[0], LJ_ERRBIT_CAPACITY);
                    atomicMax(&b.err[1], c);
                }
                longest = max(longest, c);
            }
            __syncwarp();
        }
    }
    longest = __reduce_max_sync(0xffffffffu, longest);
    if (lane == 0 && longest > 0) atomicMax(&s_longest, longest);
    __syncthreads();
    if (threadIdx.x == 0 && s_longest > 0) atomicMax(&b.err[2], s_longest);
}

// ---------------------------------------------------------------------------
// k_rebuild_cluster: binning, sort and gather of small boxes in one launch,
// by one thread-block cluster whose blocks meet at the hardware's cluster
// barrier between the stages.  A step without a build then pays two early
// exits (this and the list build) instead of five, and a build no launches
// between the stages; the list build stays a kernel of its own, as it wants
// every SM.  (A cooperative launch with grid barriers, which could hold the list
// build too, costs ~8 us inside a step graph.)  The launch rule,
// cluster_rebuild, has the times.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void cluster_barrier()
{
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

__global__ void __launch_bounds__(kClusterThreads) k_rebuild_cluster(BoxDev b, int from_abs, const int4* tiles,
                                                                      int ntiles)
{
    await_previous();
    if (!box_needs_rebuild(b)) return;   // the same word for every block: none is left waiting
    if (b.nrep > 1) {   // one replica's work is all of its own
        if (blockIdx.x == 0) phase_list_work(b);
        cluster_barrier();
    }
    phase_bin(b, from_abs);
    cluster_barrier();
    phase_scan<kClusterThreads>(b, tiles, ntiles);
    cluster_barrier();
    phase_scatter(b);
    cluster_barrier();
    phase_rank(b);
}
static_assert(kClusterThreads % LJ_CHUNK == 0, "whole groups");

}  // namespace

cudaError_t launch_bin(const BoxDev& b, int from_abs, Launch l)
{
    return launch_kernel(k_bin, l.grid, LJ_CHUNK, 0, l.s, l.early, b, from_abs);
}

cudaError_t launch_scan(const BoxDev& b, const int4* tiles, int ntiles, Launch l)
{
    return launch_kernel(k_scan, l.grid, kScanThreads, 0, l.s, l.early, b, tiles, ntiles);
}

cudaError_t launch_scatter(const BoxDev& b, Launch l)
{
    return launch_kernel(k_scatter, l.grid, LJ_CHUNK, 0, l.s, l.early, b);
}

cudaError_t launch_sortgather(const BoxDev& b, Launch l)
{
    return launch_kernel(k_sortgather, l.grid, 256, 0, l.s, l.early, b);
}

cudaError_t launch_nlist(const BoxDev& b, Launch l)
{
    const int dyn = LJ_TILE_MAX * 16;
    static bool attr = false;
    if (!attr) {
        cudaError_t e = cudaFuncSetAttribute(k_nlist, cudaFuncAttributeMaxDynamicSharedMemorySize, dyn);
        if (e != cudaSuccess) return e;
        attr = true;
    }
    k_nlist<<<l.grid, LJ_LIST_THREADS, dyn, l.s>>>(b);
    return cudaGetLastError();
}

cudaError_t launch_list_work(const BoxDev& b, unsigned long long* runs, cudaStream_t s, bool early)
{
    return launch_kernel(k_list_work, 1, 1024, 0, s, early, b, runs);
}

cudaError_t launch_nlist_lanes(const BoxDev& b, int per_particle, Launch l)
{
    const size_t dyn = (size_t)LJ_LANE_THREADS * kLaneRow * sizeof(uint32_t);   // the row buffers: below 48 KB
    return launch_kernel(per_particle == 4 ? k_nlist_lanes<4> : k_nlist_lanes<1>, l.grid, LJ_LANE_THREADS, dyn, l.s,
                         l.early, b);
}

// Whether this GPU holds the cluster (16 blocks is beyond the portable 8).
bool cluster_rebuild_fits()
{
    cudaLaunchConfig_t c{};
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = kClusterBlocks;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    c.gridDim = dim3(kClusterBlocks);
    c.blockDim = dim3(kClusterThreads);
    c.attrs = &at;
    c.numAttrs = 1;
    int n = 0;
    const bool ok =
        cudaFuncSetAttribute(k_rebuild_cluster, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess &&
        cudaOccupancyMaxActiveClusters(&n, k_rebuild_cluster, &c) == cudaSuccess && n > 0;
    if (!ok) cudaGetLastError();
    return ok;
}

cudaError_t launch_rebuild_cluster(const BoxDev& b, int from_abs, const int4* tiles, int ntiles,
                                   cudaStream_t s, bool early)
{
    cudaLaunchConfig_t c{};
    cudaLaunchAttribute at[2] = {};
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = kClusterBlocks;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[1].val.programmaticStreamSerializationAllowed = 1;
    c.gridDim = dim3(kClusterBlocks);
    c.blockDim = dim3(kClusterThreads);
    c.stream = s;
    c.attrs = at;
    c.numAttrs = early ? 2 : 1;
    return cudaLaunchKernelEx(&c, k_rebuild_cluster, b, from_abs, tiles, ntiles);
}

int ljmd_scan_tile_cells() { return kScanTile; }
