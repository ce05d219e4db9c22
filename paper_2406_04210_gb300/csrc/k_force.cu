// k_force.cu -- truncated Lennard-Jones pair force, energy and virial over the
// Verlet list (Sec. 4: Lennard-Jones pair forces; Sec. 5, Truncated Force
// Performance Study: the force kernel over Verlet lists is ~60 % of the run
// time and is memory-latency sensitive -- the CUDA version there reads packed
// float4 particle data through the texture path).
//
// The threads of particle i, in cell-sorted order, walk its list:
//   d_ij = (o_i - o_j) - shift(k)       cell-relative offsets, FP32
//   F_i += 48 eps/r^2 [(s/r)^12 - (s/r)^6/2] d_ij      for r^2 < rc^2
// E_pot and W are summed per thread in the kernel's real type, reduced per
// warp (list kernels) or per work item (all pairs) in FP64 (each pair is
// seen twice in a full list: factor 1/2).
#include "ljmd_internal.cuh"

namespace {

__device__ __forceinline__ double warp_sum_d(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    return v;
}

// Sum two doubles over the block; valid in thread 0.
__device__ __forceinline__ void block_sum2(double& a, double& c, double (*s)[32])
{
    a = warp_sum_d(a);
    c = warp_sum_d(c);
    int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (lane == 0) {
        s[0][warp] = a;
        s[1][warp] = c;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        a = 0.0;
        c = 0.0;
        for (int k = 0; k < (int)(blockDim.x >> 5); ++k) {
            a += s[0][k];
            c += s[1][k];
        }
    }
    __syncthreads();
}

// -d_ij of an FP32 pair: -d = (o_j - o_i) + (dx, dy, dz) * ell, one rounding
// for the difference and one for the shift; x and y as FP32 pairs (a gathered
// float4 holds them as a register pair).  ell is the cell edge in the digits'
// units (x, y / 4, z / 16).
__device__ __forceinline__ float2 neg_d_xy(unsigned ent, const float4& pj, const float4& pi, const float3& ell)
{
    const float2 u = __fadd2_rn(make_float2(entry_raw<0>(ent), entry_raw<1>(ent)),
                                make_float2(-digit_one(0), -digit_one(1)));
    const float2 t = __fadd2_rn(make_float2(pj.x, pj.y), make_float2(-pi.x, -pi.y));
    return __ffma2_rn(u, make_float2(ell.x, ell.y), t);
}

// One pair term of the FP32 force: accumulates f d into (fx, fy, fz) and,
// with ENERGY, the pair energy and virial; the term is masked (not branched)
// by the cutoff test, so the threads of a particle never diverge.  (The tiled
// kernel's path for a neighbourhood beyond its tile.)
template <bool MONO, bool ENERGY>
__device__ __forceinline__ void pair_f32(unsigned ent, const float4& pj, const float4& pi, int ti,
                                         const float3& ell, const float4* s_lj, const float* s_rc2,
                                         const float* s_esh, int nt, const float4& mlj, float mrc2,
                                         float mesh, float& fx, float& fy, float& fz, float& e, float& vir)
{
    const float2 dq = neg_d_xy(ent, pj, pi, ell);
    const float dz = fmaf(-entry_unit<2>(ent), ell.z, pi.z - pj.z);
    const float2 sq = __fmul2_rn(dq, dq);
    const float r2 = fmaf(dz, dz, sq.x + sq.y);
    float4 c;
    float rc2, esh;
    if (MONO) {
        c = mlj;
        rc2 = mrc2;
        esh = mesh;
    } else {
        const int pp = ti * nt + __float_as_int(pj.w);
        c = s_lj[pp];
        rc2 = s_rc2[pp];
        esh = ENERGY ? s_esh[pp] : 0.f;
    }
    const float r2i = rcp_approx(r2);
    const float r6i = r2i * r2i * r2i;
    // c = (48 eps sigma^12, 24 eps sigma^6, 4 eps sigma^12, 4 eps sigma^6)
    float f = r2i * r6i * fmaf(c.x, r6i, -c.y);
    const bool in = r2 < rc2;
    f = in ? f : 0.f;
    fx = fmaf(-f, dq.x, fx);
    fy = fmaf(-f, dq.y, fy);
    fz = fmaf(f, dz, fz);
    if (ENERGY) {
        const float u = fmaf(r6i, fmaf(c.z, r6i, -c.w), -esh);
        e += in ? u : 0.f;
        vir = fmaf(f, r2, vir);
    }
}

// Sums of k_force_f32 over a thread's pairs, in units applied at the end: 24 eps
// sigma^6 for one species, 12 for several (whose tables hold 4 eps sigma^12 and 2
// eps sigma^6).  w = sum f r^2 (the virial).  The energy needs no pair arithmetic
// of its own: with s6 = (sigma / r)^6,
//   u = 4 eps (s6^2 - s6) - shift = (f r^2) / 12 - (2 eps s6 + shift),
// so b sums the second term, in units of 2 eps sigma^6 for one species.  In
// these units it is w - b, with no constant that is rounded on its own (1/12 in
// FP32 shifts every particle's energy by 3e-8 of w / 12 alike, which the sum over
// the particles does not average out).  w and b are two partial sums each in
// pair2_f32 (its two pairs), one in pair1_f32.
// For one species f r^2 = c6 r^-6 (2 s6 - 1): the largest power formed is r^-8, so
// that the unit of length has the room it has in the tables (r^-14, in units of
// 48 eps sigma^12, is subnormal from sigma = 400 and overflows below 2e-3).
struct PairSums {
    float fx, fy, fz;
    float2 w, b;
};

// The pair constants of a particle with species 0 and with species 1 (TWO: boxes
// of two species).  Chosen by selects: the table's two shared-memory loads per
// pair share the L1 data pipe, which bounds the kernel, with the gathers.  The
// 1.2-density mixture with / without energies, table -> selects: N = 256,000
// 74.3 / 67.9 -> 64.0 / 59.3 us, 1M 241 / 217 -> 208 / 189, 32,000 20.7 / 18.2
// -> 18.4 / 17.0.  The row's ten constants take registers: five blocks of 256
// per SM with energies (six: 1M 223 us), six without.
struct RowConsts {
    float4 c0, c1;   // 4 eps sigma^12, -2 eps sigma^6, 2 eps sigma^6, shift
    float r0, r1;    // rc^2
};

// Two pair terms: the separations one by one, everything from r^2 on as FP32
// pairs.  The cutoff masks 1/r^2 (times 1 or 0), so that every term of a pair
// beyond it, the sentinel's too, is 0.
template <bool MONO, bool ENERGY, bool TWO>
__device__ __forceinline__ void pair2_f32(unsigned e0, const float4& q0, unsigned e1, const float4& q1,
                                          const float4& pi, int tb, const float3& ell, const float4* s_lj,
                                          const float* s_rc2, float tw, float kap, float mrc2, const RowConsts& rc,
                                          PairSums& S)
{
    const float2 a0 = neg_d_xy(e0, q0, pi, ell), a1 = neg_d_xy(e1, q1, pi, ell);
    const float2 az = make_float2(fmaf(entry_unit<2>(e0), ell.z, q0.z - pi.z), fmaf(entry_unit<2>(e1), ell.z, q1.z - pi.z));
    const float2 s0 = __fmul2_rn(a0, a0), s1 = __fmul2_rn(a1, a1);
    const float2 r2 = __ffma2_rn(az, az, make_float2(s0.x + s0.y, s1.x + s1.y));
    float2 c12, nc6, rc2, hb, esh;
    if (MONO) {
        c12 = make_float2(tw, tw);
        nc6 = make_float2(-1.f, -1.f);
        rc2 = make_float2(mrc2, mrc2);
    } else {
        const int p0 = tb + __float_as_int(q0.w), p1 = tb + __float_as_int(q1.w);
        const float4 c0 = TWO ? (p0 & 1 ? rc.c1 : rc.c0) : s_lj[p0], c1 = TWO ? (p1 & 1 ? rc.c1 : rc.c0) : s_lj[p1];
        c12 = make_float2(c0.x, c1.x);
        nc6 = make_float2(c0.y, c1.y);
        hb = make_float2(c0.z, c1.z);
        esh = make_float2(c0.w, c1.w);
        rc2 = TWO ? make_float2(p0 & 1 ? rc.r1 : rc.r0, p1 & 1 ? rc.r1 : rc.r0) : make_float2(s_rc2[p0], s_rc2[p1]);
    }
    const float2 in = make_float2(r2.x < rc2.x ? 1.f : 0.f, r2.y < rc2.y ? 1.f : 0.f);
    const float2 ri = __fmul2_rn(make_float2(rcp_approx(r2.x), rcp_approx(r2.y)), in);
    const float2 r6 = __fmul2_rn(__fmul2_rn(ri, ri), ri);
    const float2 g = __fmul2_rn(r6, __ffma2_rn(c12, r6, nc6));   // f r^2
    const float2 f = __fmul2_rn(ri, g);
    S.fx = fmaf(f.x, a0.x, S.fx);   // of -d: the sums are negated at the end
    S.fy = fmaf(f.x, a0.y, S.fy);
    S.fz = fmaf(f.x, az.x, S.fz);
    S.fx = fmaf(f.y, a1.x, S.fx);
    S.fy = fmaf(f.y, a1.y, S.fy);
    S.fz = fmaf(f.y, az.y, S.fz);
    if (ENERGY) {
        S.w = __fadd2_rn(S.w, g);
        if (MONO) S.b = __fadd2_rn(S.b, __ffma2_rn(in, make_float2(kap, kap), r6));
        else S.b = __ffma2_rn(esh, in, __ffma2_rn(hb, r6, S.b));
    }
}

// One pair term, the same sums, in scalar arithmetic: more instructions, but it
// fits the 32 registers of eight blocks of 256 per SM (packed operands and
// constants take register pairs).
template <bool MONO, bool ENERGY, bool TWO>
__device__ __forceinline__ void pair1_f32(unsigned e0, const float4& q0, const float4& pi, int tb, const float3& ell,
                                          const float4* s_lj, const float* s_rc2, float tw, float kap, float mrc2,
                                          const RowConsts& rc, PairSums& S)
{
    const float2 a0 = neg_d_xy(e0, q0, pi, ell);
    const float az = fmaf(entry_unit<2>(e0), ell.z, q0.z - pi.z);
    const float2 s0 = __fmul2_rn(a0, a0);
    const float r2 = fmaf(az, az, s0.x + s0.y);
    float4 c = make_float4(0.f, 0.f, 0.f, 0.f);
    float rc2 = mrc2;
    if (!MONO) {
        const int p0 = tb + __float_as_int(q0.w);
        if (TWO) {   // tb is even
            const bool o = __float_as_int(q0.w) != 0;
            c = make_float4(o ? rc.c1.x : rc.c0.x, o ? rc.c1.y : rc.c0.y, o ? rc.c1.z : rc.c0.z, o ? rc.c1.w : rc.c0.w);
            rc2 = o ? rc.r1 : rc.r0;
        } else {
            c = s_lj[p0];
            rc2 = s_rc2[p0];
        }
    }
    const bool in = r2 < rc2;
    const float ri = in ? rcp_approx(r2) : 0.f;
    const float r6 = ri * ri * ri;
    const float g = MONO ? fmaf(tw * r6, r6, -r6) : r6 * fmaf(c.x, r6, c.y);   // f r^2
    const float f = ri * g;
    S.fx = fmaf(f, a0.x, S.fx);   // of -d: the sums are negated at the end
    S.fy = fmaf(f, a0.y, S.fy);
    S.fz = fmaf(f, az, S.fz);
    if (ENERGY) {
        S.w.x += g;
        if (MONO) S.b.x += r6 + (in ? kap : 0.f);
        else S.b.x = fmaf(c.z, r6, S.b.x + (in ? c.w : 0.f));
    }
}

// FP32 pair force (Sec. 4/5), LJ_TPP (4) threads per particle.  A particle's
// row is read in blocks of LJ_ROW_BLOCK (16) entries, the last block's entries
// past the count replaced by the sentinel slot; each thread takes four
// consecutive entries of a block with one 16-byte load (the next block's load
// in flight while this one is computed) and gathers the four neighbours' FP32
// offsets through L1 (four gathers in flight); the four threads combine their
// partial forces with shuffles.
// Work items: chunks of 128 particles, two passes of 64 by a block of 256; or,
// SPREAD, 16 particles by a block of 64 threads (the rule is at spread_force).
// What bounds it.  Chunks: the L1 data pipe, ~10 wavefronts per gather (67 %
// of peak over the launch, 79 % while active), which neither fewer
// instructions (33.4 M -> 26.5 M with the packed pairs: 47.2 us against 45.6
// at 256k, fewer resident warps), nor rows in the order of slot mod 8 (fewer
// bank conflicts, more lines: 44.7 us, but 662 us against 588 at 4M) moved, so
// resident warps matter most: 32 registers and eight blocks per SM for one
// species, 40 and six for several (two: see RowConsts).  With the digits below the slot and the
// energy from sums the force needs anyway: 4M with energies 589 -> 573 us,
// without 529 -> 515, the 256k mixture 78.6 -> 75.3.  SPREAD: the serial row
// (five dependent blocks), on every SM instead of a few: N = 4,000 16.4 -> 9.0
// us, N = 32,000 17.2 -> 12.8 us; packed pairs, as registers are free there.
// MONO: a single species, its pair constants read from the kernel
// parameters.  SINGLE (MONO and one replica): the cell edge from the
// parameters too.  One (E_pot, W) share per warp and item.
static_assert(LJ_TPP * 4 == LJ_ROW_BLOCK, "a row block is one 16-byte load per thread of a particle");
template <bool MONO, bool ENERGY, bool SINGLE, int THREADS, int RES, bool TWO = false>
__global__ void __launch_bounds__(THREADS, RES) k_force_f32(BoxDev b)
{
    await_previous();
    constexpr int TPP = LJ_TPP;
    constexpr bool SPREAD = THREADS == LJ_SPREAD_THREADS;
    constexpr int PASS = THREADS / TPP;                       // particles of a pass
    constexpr int PARTS = SPREAD ? LJ_CHUNK / PASS : 1;       // work items of a chunk
    constexpr int OWN = LJ_CHUNK / PARTS;                     // particles of an item
    __shared__ float4 s_lj[MONO ? 1 : LJ_MAXT * LJ_MAXT];     // 4 eps sigma^12, -2 eps sigma^6, 2 eps sigma^6, shift
    __shared__ float s_rc2[MONO ? 1 : LJ_MAXT * LJ_MAXT];
    if (!MONO) {
        const LJDev* lj = b.lj;
        for (int k = threadIdx.x; k < b.nt * b.nt; k += blockDim.x) {
            s_lj[k] = make_float4(lj->e12[k], -0.5f * lj->e6[k], 0.5f * lj->e6[k], lj->shift[k]);
            s_rc2[k] = lj->rc2[k];
        }
        __syncthreads();   // the pair tables are complete (the block's only barrier)
    }
    // one species: f r^2 = c6 r6 (tw r6 - 1), the energy's second term (e6 / 2) (r6 + kap)
    const float unit = MONO ? b.c1.y : 12.f, eunit = MONO ? 0.5f * b.c1.w : 1.f, tw = b.tw_1, kap = b.kap_1, mrc2 = b.rc2_1;
    const int K = b.K;
    const int grp = threadIdx.x / TPP, lt = threadIdx.x % TPP;
    const float4* posq = b.posq;
    const unsigned sent = entry_make(13, b.np);
    int cur_r = -1;
    float3 ell = make_float3(b.ell1.x, 0.25f * b.ell1.y, 0.0625f * b.ell1.z);   // edges in the digits' units
    for (int it = blockIdx.x; it < b.nchunk * PARTS; it += gridDim.x) {
        const int w = it / PARTS, part = it % PARTS;
        const int4 ch = chunk_of(b, w);
        const int r = ch.x;
        if (!SINGLE && r != cur_r) {            // block-uniform
            const RepDev& R = b.rep[r];
            ell = make_float3(R.ellf[0], 0.25f * R.ellf[1], 0.0625f * R.ellf[2]);
            cur_r = r;
        }
        if (threadIdx.x == 0 && part == 0) {
            if (w == 0) *b.any_req = 0;         // the list update of this step has run
            if (b.nrep == 1 ? w == 0 : w == b.rep[r].chunk_off) {      // clear the replica's rebuild triggers
                b.disp_max[r] = 0u;
                b.rebuild_req[r] = 0;
            }
        }
        PairSums S;
        S.w = S.b = make_float2(0.f, 0.f);
        const int first = ch.y + part * OWN, last = min(first + OWN, ch.z);
        for (int base = first; base < last; base += PASS) {
            const int p = base + grp;
            const bool act = p < last;
            float4 pi = make_float4(0.f, 0.f, 0.f, 0.f);
            int cnt = 0;
            const uint4* L = reinterpret_cast<const uint4*>(b.nbr + (size_t)K * p) + lt;
            uint4 cur = make_uint4(0u, 0u, 0u, 0u);
            if (act) {
                pi = posq[p];
                cnt = min(b.nbr_count[p], K);
                cur = __ldcs(L);   // the row's first block (K >= 16 slots), in flight with the count
            }
            const int nblk = (cnt + 4 * TPP - 1) / (4 * TPP);
            const int tb = MONO ? 0 : __float_as_int(pi.w) * b.nt;
            RowConsts rc;
            if (TWO) {
                rc.c0 = s_lj[tb];
                rc.c1 = s_lj[tb + 1];
                rc.r0 = s_rc2[tb];
                rc.r1 = s_rc2[tb + 1];
            }
            S.fx = S.fy = S.fz = 0.f;
            // four entries: four gathers in flight
            auto block4 = [&](const uint4& q) {
                const float4 p0 = posq[entry_slot(q.x)];
                const float4 p1 = posq[entry_slot(q.y)];
                const float4 p2 = posq[entry_slot(q.z)];
                const float4 p3 = posq[entry_slot(q.w)];
                if (SPREAD) {
                    pair2_f32<MONO, ENERGY, TWO>(q.x, p0, q.y, p1, pi, tb, ell, s_lj, s_rc2, tw, kap, mrc2, rc, S);
                    pair2_f32<MONO, ENERGY, TWO>(q.z, p2, q.w, p3, pi, tb, ell, s_lj, s_rc2, tw, kap, mrc2, rc, S);
                } else {
                    pair1_f32<MONO, ENERGY, TWO>(q.x, p0, pi, tb, ell, s_lj, s_rc2, tw, kap, mrc2, rc, S);
                    pair1_f32<MONO, ENERGY, TWO>(q.y, p1, pi, tb, ell, s_lj, s_rc2, tw, kap, mrc2, rc, S);
                    pair1_f32<MONO, ENERGY, TWO>(q.z, p2, pi, tb, ell, s_lj, s_rc2, tw, kap, mrc2, rc, S);
                    pair1_f32<MONO, ENERGY, TWO>(q.w, p3, pi, tb, ell, s_lj, s_rc2, tw, kap, mrc2, rc, S);
                }
            };
            if (nblk > 0) {
                for (int blk = 1; blk < nblk; ++blk) {
                    const uint4 nxt = __ldcs(L + blk * TPP);   // in flight during this block
                    block4(cur);
                    cur = nxt;
                }
                // the row's last block: entries past the count (stale or
                // never written) name the sentinel slot
                const int lim = cnt - ((nblk - 1) * 4 * TPP + 4 * lt);
                cur.x = lim > 0 ? cur.x : sent;
                cur.y = lim > 1 ? cur.y : sent;
                cur.z = lim > 2 ? cur.z : sent;
                cur.w = lim > 3 ? cur.w : sent;
                block4(cur);
            }
#pragma unroll
            for (int o = TPP / 2; o > 0; o >>= 1) {
                S.fx += __shfl_xor_sync(0xffffffffu, S.fx, o);
                S.fy += __shfl_xor_sync(0xffffffffu, S.fy, o);
                S.fz += __shfl_xor_sync(0xffffffffu, S.fz, o);
            }
            if (act && lt == 0) {
                b.force4[p] = make_float4(-unit * S.fx, -unit * S.fy, -unit * S.fz, 0.f);
                if (!isfinite(S.fx + S.fy + S.fz)) atomicOr(&b.err[0], LJ_ERRBIT_NONFINITE);
            }
        }
        if (ENERGY) {
            // one (E_pot, W) share per warp and item, no block barrier: the
            // warps of a block run ahead into the next item independently.
            // The warp sum is double-single (two FP32 words per partial
            // sum): FP64-class precision on the FP32 pipe, since FP64 adds
            // are scarce on this GPU.  The share is stored as the (hi, lo)
            // pair itself (pf_ds), halved exactly; the reduction converts
            const float w = S.w.x + S.w.y, vir = unit * w;
            const float e = eunit * (w - (S.b.x + S.b.y));
            const float2 d = warp_sum2_ds2(e, vir);
            if ((threadIdx.x & 15) == 0) {
                const size_t q = (size_t)it * (THREADS / 16) + (threadIdx.x >> 4);
                reinterpret_cast<float2*>(b.part_f)[q] = make_float2(0.5f * d.x, 0.5f * d.y);
            }
        }
    }
}

// ---------------------------------------------------------------------------
// Tiled FP32 pair force (Sec. 4/5: the same forces, energy and virial as
// k_force_f32; Sec. 5 finds the force kernel bound by fetching neighbour
// data, which here comes from shared memory).  The work items are bricks
// of up to 2 x 2 x 2 cells.  A producer warp stages the FP32 offsets of a
// brick's neighbourhood (its cells and the layer of cells around them, up to
// 64 cells) as x, y and z planes of a shared-memory tile, each moved into
// the frame of the brick's centre by one FMA (q_j = o_j + a ell, a a
// multiple of 1/2, one rounding), double-buffered; the consumer warps walk
// the brick's particles' list rows, LJ_TPP threads per particle, four
// entries per thread and 16-entry row block.  An entry (stencil digits of neighbour cell k, slot j) names the
// tile element j - start + base of the tile cell at the particle's cell plus
// k: its byte address is (entry >> 4) plus a table word of the particle's
// cell indexed by the digits, which also cancels what the shift leaves of
// the digits -- one shift-add per entry, no decode and no image shift per
// pair.  Pairs are evaluated two at a time with FP32-pair arithmetic on
// d' = q_j - p_i = -d_ij (p_i = o_i + a_i ell, the sums negated at the
// end).  Brick edges are 2 cells only where a tile coordinate stays below 8
// (one rounding of 2^-22 at most); a brick whose neighbourhood holds more
// than LJ_BRICK_TILE particles is evaluated from global memory as in
// k_force_f32.  Energy and virial: one double-single (E_pot, W) share per
// warp and brick, summed in FP64 by k_thermo in a fixed order.
// ---------------------------------------------------------------------------

// x, y, z of the tile element at byte address a (planes PL bytes apart)
template <int PL>
__device__ __forceinline__ void tile_xyz(uint32_t a, float& x, float& y, float& z)
{
    asm("ld.shared.f32 %0, [%3];\n\t"
        "ld.shared.f32 %1, [%3+%4];\n\t"
        "ld.shared.f32 %2, [%3+%5];"
        : "=f"(x), "=f"(y), "=f"(z)
        : "r"(a), "n"(PL), "n"(2 * PL));
}
template <int PL>
__device__ __forceinline__ int tile_type(uint32_t a)
{
    int t;
    asm("ld.shared.b32 %0, [%1+%2];" : "=r"(t) : "r"(a), "n"(3 * PL));
    return t;
}

struct PairAcc2 {
    float2 fx, fy, fz, e, w;
};

// Two pair terms (tile elements at a0, a1) against particle i (n = -p_i),
// accumulated as FP32 pairs; masked, not branched, by the cutoff test.
template <bool MONO, bool ENERGY, int PL>
__device__ __forceinline__ void tile_pair2(uint32_t a0, uint32_t a1, const float2& nx, const float2& ny,
                                           const float2& nz, int ti, int nt, const float4* s_lj,
                                           const float* s_rc2, const float* s_esh, const float4& mlj,
                                           float mrc2, float mesh, PairAcc2& A)
{
    float x0, y0, z0, x1, y1, z1;
    tile_xyz<PL>(a0, x0, y0, z0);
    tile_xyz<PL>(a1, x1, y1, z1);
    const float2 dx = __fadd2_rn(make_float2(x0, x1), nx);
    const float2 dy = __fadd2_rn(make_float2(y0, y1), ny);
    const float2 dz = __fadd2_rn(make_float2(z0, z1), nz);
    const float2 r2 = __ffma2_rn(dz, dz, __ffma2_rn(dy, dy, __fmul2_rn(dx, dx)));
    float2 c12, nc6, e12, ne6, rc2, nesh;
    if (MONO) {
        c12 = make_float2(mlj.x, mlj.x);
        nc6 = make_float2(-mlj.y, -mlj.y);
        e12 = make_float2(mlj.z, mlj.z);
        ne6 = make_float2(-mlj.w, -mlj.w);
        rc2 = make_float2(mrc2, mrc2);
        nesh = make_float2(-mesh, -mesh);
    } else {
        const int p0 = ti * nt + tile_type<PL>(a0), p1 = ti * nt + tile_type<PL>(a1);
        const float4 q0 = s_lj[p0], q1 = s_lj[p1];
        c12 = make_float2(q0.x, q1.x);
        nc6 = make_float2(-q0.y, -q1.y);
        e12 = make_float2(q0.z, q1.z);
        ne6 = make_float2(-q0.w, -q1.w);
        rc2 = make_float2(s_rc2[p0], s_rc2[p1]);
        nesh = ENERGY ? make_float2(-s_esh[p0], -s_esh[p1]) : make_float2(0.f, 0.f);
    }
    const float2 ri = make_float2(rcp_approx(r2.x), rcp_approx(r2.y));
    const float2 r6 = __fmul2_rn(__fmul2_rn(ri, ri), ri);
    float2 f = __fmul2_rn(__fmul2_rn(ri, r6), __ffma2_rn(c12, r6, nc6));
    const bool in0 = r2.x < rc2.x, in1 = r2.y < rc2.y;
    f.x = in0 ? f.x : 0.f;
    f.y = in1 ? f.y : 0.f;
    A.fx = __ffma2_rn(f, dx, A.fx);
    A.fy = __ffma2_rn(f, dy, A.fy);
    A.fz = __ffma2_rn(f, dz, A.fz);
    if (ENERGY) {
        float2 u = __ffma2_rn(r6, __ffma2_rn(e12, r6, ne6), nesh);
        u.x = in0 ? u.x : 0.f;
        u.y = in1 ? u.y : 0.f;
        A.e = __fadd2_rn(A.e, u);
        A.w = __ffma2_rn(f, r2, A.w);
    }
}

// tile address of entry e for the particle's address table D
__device__ __forceinline__ uint32_t tile_addr(uint32_t e, const uint32_t* D) { return (e >> 4) + D[e & 63u]; }

static_assert(LJ_BRICK_WARPS == LJ_FORCE_WARPS, "per-brick shares in the chunk kernel's share stride");
constexpr int kBrickThreads = LJ_BRICK_THREADS;          // consumer threads
constexpr int kBrickWarps = kBrickThreads / 32;          // consumer warps (the producer is warp kBrickWarps)
constexpr int kBrickPass = kBrickThreads / LJ_TPP;       // particles per consumer pass

__device__ __forceinline__ void mbar_arrive1(unsigned long long* bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

// Dynamic shared memory of k_force_tile_f32: two buffers of NPL planes.
constexpr size_t tile_buf_bytes(bool mono) { return (size_t)(mono ? 3 : 4) * (LJ_BRICK_TILE + 1) * 4; }

// Producer warp kBrickWarps stages brick k + 1 (tile planes, brick-cell
// tables, address tables) into one buffer while the consumer warps compute
// brick k from the other; full[buf] (32 arrivals, the producer's lanes) and
// empty[buf] (kBrickThreads arrivals, the consumers) hand the buffers over.
// Every wait is bounded: on a timeout the warp records LJ_ERRBIT_TIMEOUT and
// leaves, and the others then time out in turn.
template <bool MONO, bool ENERGY>
__global__ void __launch_bounds__(LJ_BRICK_THREADS + 32, 4) k_force_tile_f32(BoxDev b)
{
    constexpr int T = LJ_BRICK_TILE;
    constexpr int NPL = MONO ? 3 : 4;   // x, y, z (and type) planes
    constexpr int PL = (T + 1) * 4;     // bytes per plane; element T of each is the sentinel
    constexpr int BUF = NPL * PL;       // bytes per buffer
    constexpr unsigned FULL = 0xffffffffu;
    extern __shared__ __align__(16) float s_dyn[];   // [2][NPL][T + 1]
    __shared__ uint32_t s_D[2][8][64];  // per buffer, brick cell and stencil-digit code: tile address term
    __shared__ int s_pc[2][9], s_cs[2][8], s_nb[2], s_tiled[2];   // per buffer: brick cells, particles
    __shared__ int s_tb[64], s_ts[64], s_tn[64];                  // producer: tile cells
    __shared__ unsigned long long s_full[2], s_empty[2];
    __shared__ float4 s_lj[MONO ? 1 : LJ_MAXT * LJ_MAXT];
    __shared__ float s_rc2[MONO ? 1 : LJ_MAXT * LJ_MAXT];
    __shared__ float s_esh[MONO ? 1 : LJ_MAXT * LJ_MAXT];
    const int nt = b.nt;
    if (!MONO) {
        const LJDev* lj = b.lj;
        for (int k = threadIdx.x; k < nt * nt; k += blockDim.x) {
            s_lj[k] = make_float4(lj->c12[k], lj->c6[k], lj->e12[k], lj->e6[k]);
            s_rc2[k] = lj->rc2[k];
            s_esh[k] = lj->shift[k];
        }
    }
    if (threadIdx.x < 2 * NPL) {   // sentinels: far offsets, type 0
        const int q = threadIdx.x % NPL;
        s_dyn[(threadIdx.x / NPL) * NPL * (T + 1) + q * (T + 1) + T] = q < 3 ? LJ_SENTINEL_OFF : 0.f;
    }
    if (threadIdx.x == 0) {
        mbar_init(&s_full[0], 32);
        mbar_init(&s_full[1], 32);
        mbar_init(&s_empty[0], kBrickThreads);
        mbar_init(&s_empty[1], kBrickThreads);
    }
    __syncthreads();   // the block's only barrier: the roles part here
    const uint32_t X0 = (uint32_t)__cvta_generic_to_shared(s_dyn);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const float4* posq = b.posq;

    if (warp == kBrickWarps) {
        // ---------------- producer ----------------
        int k = 0;
        for (int bi = blockIdx.x; bi < b.nbrick; bi += gridDim.x, ++k) {
            const int buf = k & 1;
            if (k >= 2 && !mbar_wait(&s_empty[buf], ((k >> 1) - 1) & 1)) {
                if (lane == 0) atomicOr(&b.err[0], LJ_ERRBIT_TIMEOUT);
                return;
            }
            const int4 B = b.brick[bi];
            const int r = B.x;
            const RepDev& R = b.rep[r];
            if (lane == 0) {
                if (bi == 0) *b.any_req = 0;   // the list update of this step has run
                if (B.y == 0 && B.z == 0 && B.w == 0) {   // the replica's first brick: clear its rebuild triggers
                    b.disp_max[r] = 0u;
                    b.rebuild_req[r] = 0;
                }
            }
            const int ex = min(R.br[0], R.nc[0] - B.y), ey = min(R.br[1], R.nc[1] - B.z),
                      ez = min(R.br[2], R.nc[2] - B.w);
            const int tx = ex + 2, txy = tx * (ey + 2), ntc = txy * (ez + 2), nbc = ex * ey * ez;
            const int sx = ex - 1, sy = ey - 1;   // brick cell cl = u + ex (v + ey w): u = cl & sx, ...
            const float3 ell = make_float3(R.ellf[0], R.ellf[1], R.ellf[2]);
            // tile coordinate t along an axis (brick cell u is t = u + 1): its
            // offset in cells from the brick centre, t - (extent + 1) / 2
            const float hx = 0.5f * (float)(ex + 1), hy = 0.5f * (float)(ey + 1), hz = 0.5f * (float)(ez + 1);
            // tile cells 2 lane and 2 lane + 1: first slot and particles, then
            // their bases (exclusive prefix over the tile)
            int js[2] = {0, 0}, nk[2] = {0, 0};
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const int t = 2 * lane + u;
                if (t < ntc) {
                    const int a = t % tx, c = t / txy, bb = (t / tx) - c * (ey + 2);
                    const int cn = R.cell_off + wrapi(B.y - 1 + a, R.nc[0]) +
                                   R.nc[0] * (wrapi(B.z - 1 + bb, R.nc[1]) + R.nc[1] * wrapi(B.w - 1 + c, R.nc[2]));
                    js[u] = b.cell_start[cn];
                    nk[u] = b.cell_end[cn] - js[u];
                }
            }
            int incl = nk[0] + nk[1];
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int t = __shfl_up_sync(FULL, incl, o);
                if (lane >= o) incl += t;
            }
            const int e0 = incl - nk[0] - nk[1];
            s_tb[2 * lane] = e0;
            s_tb[2 * lane + 1] = e0 + nk[0];
            s_ts[2 * lane] = js[0];
            s_ts[2 * lane + 1] = js[1];
            s_tn[2 * lane] = nk[0];
            s_tn[2 * lane + 1] = nk[1];
            const bool tiled = __shfl_sync(FULL, incl, 31) <= T;
            __syncwarp();
            // brick cells (lane < 8): first slot and particle prefix
            int n8 = 0;
            if (lane < nbc) {
                const int u = lane & sx, v = (lane >> sx) & sy, w = lane >> (sx + sy);
                const int t = (u + 1) + tx * (v + 1) + txy * (w + 1);
                s_cs[buf][lane] = s_ts[t];
                n8 = s_tn[t];
            }
            int inc8 = n8;
#pragma unroll
            for (int o = 1; o < 8; o <<= 1) {
                const int t = __shfl_up_sync(FULL, inc8, o);
                if (lane >= o) inc8 += t;
            }
            if (lane < 8) s_pc[buf][lane + 1] = inc8;   // lanes past the brick's cells add nothing
            const int npb = __shfl_sync(FULL, inc8, 7);
            if (lane == 0) {
                s_pc[buf][0] = 0;
                s_nb[buf] = npb;
                s_tiled[buf] = tiled ? 1 : 0;
            }
            if (tiled) {
                float* const P = s_dyn + buf * NPL * (T + 1);
                const uint32_t Xb = X0 + (uint32_t)(buf * BUF);
                // rows of the tile (tile cells along x at one y, z), 4 elements
                // per lane in flight
                const int nrow = (ey + 2) * (ez + 2);
                for (int rr = 0; rr < nrow; ++rr) {
                    const int t0 = rr * tx;
                    const int rb = s_tb[t0], re = s_tb[t0 + tx - 1] + s_tn[t0 + tx - 1];
                    const float ay = (float)(rr % (ey + 2)) - hy, az = (float)(rr / (ey + 2)) - hz;   // exact
                    for (int f0 = rb; f0 < re; f0 += 128) {
                        float4 v[4];
                        int at[4];
#pragma unroll
                        for (int u = 0; u < 4; ++u) {
                            const int e = f0 + 32 * u + lane;
                            int a = 0;   // the tile cell of element e along the row
#pragma unroll
                            for (int c = 1; c < 4; ++c) a += (c < tx && s_tb[t0 + c] <= e) ? 1 : 0;
                            at[u] = a;
                            v[u] = e < re ? posq[s_ts[t0 + a] + (e - s_tb[t0 + a])] : make_float4(0.f, 0.f, 0.f, 0.f);
                        }
#pragma unroll
                        for (int u = 0; u < 4; ++u) {
                            const int e = f0 + 32 * u + lane;
                            if (e < re) {
                                P[e] = fmaf((float)at[u] - hx, ell.x, v[u].x);
                                P[(T + 1) + e] = fmaf(ay, ell.y, v[u].y);
                                P[2 * (T + 1) + e] = fmaf(az, ell.z, v[u].z);
                                if (!MONO) P[(NPL - 1) * (T + 1) + e] = v[u].w;   // type bits
                            }
                        }
                    }
                }
                // address tables: brick cell cl, stencil cell k
                for (int t = lane; t < nbc * 27; t += 32) {
                    const int cl = t / 27, kk = t - 27 * cl;
                    const int u = cl & sx, v = (cl >> sx) & sy, w = cl >> (sx + sy);
                    const uint32_t dxd = kk % 3, dyd = (kk / 3) % 3, dzd = kk / 9;
                    const int tc = (u + (int)dxd) + tx * (v + (int)dyd) + txy * (w + (int)dzd);
                    // (entry >> 4) = 4 j + dz digit
                    s_D[buf][cl][(dzd << 4) | (dyd << 2) | dxd] = Xb + 4u * (uint32_t)(s_tb[tc] - s_ts[tc]) - dzd;
                }
            }
            mbar_arrive1(&s_full[buf]);   // every producer lane: its stores precede the arrival
        }
        return;
    }

    // ---------------- consumers ----------------
    const int grp = threadIdx.x / LJ_TPP, l4 = threadIdx.x % LJ_TPP;
    const int K = b.K;
    const float4 mlj = b.c1;
    const float mrc2 = b.rc2_1, mesh = b.esh_1;
    const unsigned sent_ent = entry_make(13, b.np);
    int k = 0;
    for (int bi = blockIdx.x; bi < b.nbrick; bi += gridDim.x, ++k) {
        const int buf = k & 1;
        if (!mbar_wait(&s_full[buf], (k >> 1) & 1)) {
            if (lane == 0) atomicOr(&b.err[0], LJ_ERRBIT_TIMEOUT);
            return;
        }
        const int4 B = b.brick[bi];
        const RepDev& R = b.rep[B.x];
        const int ex = min(R.br[0], R.nc[0] - B.y), ey = min(R.br[1], R.nc[1] - B.z),
                  ez = min(R.br[2], R.nc[2] - B.w);
        const int nbc = ex * ey * ez, sx = ex - 1, sy = ey - 1;
        const float3 ell = make_float3(R.ellf[0], R.ellf[1], R.ellf[2]);
        const float hx = 0.5f * (float)(ex + 1), hy = 0.5f * (float)(ey + 1), hz = 0.5f * (float)(ez + 1);
        const bool tiled = s_tiled[buf] != 0;
        const int npb = s_nb[buf];
        const uint32_t SENT = X0 + (uint32_t)(buf * BUF) + 4u * (uint32_t)T;
        float e_acc = 0.f, w_acc = 0.f;   // this thread's energy and virial over the brick
        for (int ib = 0; ib < npb; ib += kBrickPass) {
            if (ib + (32 / LJ_TPP) * warp >= npb) break;   // warp-uniform: none of its particles here or later
            const int slot = ib + grp;
            const bool act = slot < npb;
            // its brick cell: the last cl < nbc with s_pc[cl] <= slot (prefix non-decreasing)
            const int* pc = s_pc[buf];
            int cl = (4 < nbc && pc[4] <= slot) ? 4 : 0;
            cl += (cl + 2 < nbc && pc[cl + 2] <= slot) ? 2 : 0;
            cl += (cl + 1 < nbc && pc[cl + 1] <= slot) ? 1 : 0;
            const int p = act ? s_cs[buf][cl] + (slot - pc[cl]) : 0;   // no load for an idle group
            const float4 pi = act ? posq[p] : make_float4(0.f, 0.f, 0.f, 0.f);
            const uint4* L = reinterpret_cast<const uint4*>(b.nbr + (size_t)K * p) + l4;
            const uint4 z4 = make_uint4(0u, 0u, 0u, 0u);
            // the row's first two blocks (inside the row's K >= 16 slots), in
            // flight with the count; later blocks two ahead
            uint4 cur = act ? __ldcs(L) : z4;
            uint4 nx1 = act && K > LJ_ROW_BLOCK ? __ldcs(L + LJ_TPP) : z4;
            const int cnt = act ? min(b.nbr_count[p], K) : 0;
            const int nblk = (cnt + LJ_ROW_BLOCK - 1) / LJ_ROW_BLOCK;
            const int ti = __float_as_int(pi.w);
            const int lim = cnt - ((nblk - 1) * LJ_ROW_BLOCK + 4 * l4);   // valid entries of the last block
            PairAcc2 A;
            A.fx = A.fy = A.fz = A.e = A.w = make_float2(0.f, 0.f);
            if (tiled) {
                const int u = cl & sx, v = (cl >> sx) & sy, w = cl >> (sx + sy);
                // p_i in the brick frame: one rounding
                const float px = fmaf((float)(u + 1) - hx, ell.x, pi.x), py = fmaf((float)(v + 1) - hy, ell.y, pi.y),
                            pz = fmaf((float)(w + 1) - hz, ell.z, pi.z);
                const float2 nx = make_float2(-px, -px), ny = make_float2(-py, -py), nz = make_float2(-pz, -pz);
                const uint32_t* D = s_D[buf][cl];
                for (int blk = 0; blk + 1 < nblk; ++blk) {
                    const uint4 nx2 = blk + 2 < nblk ? __ldcs(L + (blk + 2) * LJ_TPP) : z4;   // two ahead
                    tile_pair2<MONO, ENERGY, PL>(tile_addr(cur.x, D), tile_addr(cur.y, D), nx, ny, nz, ti, nt, s_lj,
                                                 s_rc2, s_esh, mlj, mrc2, mesh, A);
                    tile_pair2<MONO, ENERGY, PL>(tile_addr(cur.z, D), tile_addr(cur.w, D), nx, ny, nz, ti, nt, s_lj,
                                                 s_rc2, s_esh, mlj, mrc2, mesh, A);
                    cur = nx1;
                    nx1 = nx2;
                }
                if (nblk > 0) {   // the last block: entries past the count name the sentinel
                    const uint32_t a0 = lim > 0 ? tile_addr(cur.x, D) : SENT;
                    const uint32_t a1 = lim > 1 ? tile_addr(cur.y, D) : SENT;
                    const uint32_t a2 = lim > 2 ? tile_addr(cur.z, D) : SENT;
                    const uint32_t a3 = lim > 3 ? tile_addr(cur.w, D) : SENT;
                    tile_pair2<MONO, ENERGY, PL>(a0, a1, nx, ny, nz, ti, nt, s_lj, s_rc2, s_esh, mlj, mrc2, mesh, A);
                    tile_pair2<MONO, ENERGY, PL>(a2, a3, nx, ny, nz, ti, nt, s_lj, s_rc2, s_esh, mlj, mrc2, mesh, A);
                }
            } else {   // neighbourhood larger than the tile: gathers from global memory
                const float3 ell_digit = make_float3(ell.x, 0.25f * ell.y, 0.0625f * ell.z);
                float fx = 0.f, fy = 0.f, fz = 0.f, e = 0.f, vir = 0.f;
                for (int blk = 0; blk < nblk; ++blk) {
                    const bool last = blk + 1 == nblk;
                    const uint4 nx2 = blk + 2 < nblk ? __ldcs(L + (blk + 2) * LJ_TPP) : z4;
                    uint32_t q[4] = {cur.x, cur.y, cur.z, cur.w};
#pragma unroll
                    for (int kk = 0; kk < 4; ++kk) {
                        const unsigned ek = (!last || lim > kk) ? q[kk] : sent_ent;
                        const float4 pj = posq[entry_slot(ek)];
                        pair_f32<MONO, ENERGY>(ek, pj, pi, ti, ell_digit, s_lj, s_rc2, s_esh, nt, mlj, mrc2, mesh, fx,
                                               fy, fz, e, vir);
                    }
                    cur = nx1;
                    nx1 = nx2;
                }
                // d_ij orientation here: stored negated like the tile path's sums
                A.fx = make_float2(-fx, 0.f);
                A.fy = make_float2(-fy, 0.f);
                A.fz = make_float2(-fz, 0.f);
                A.e = make_float2(e, 0.f);
                A.w = make_float2(vir, 0.f);
            }
            float fx = A.fx.x + A.fx.y, fy = A.fy.x + A.fy.y, fz = A.fz.x + A.fz.y;
            if (ENERGY) {   // idle groups hold zeros
                e_acc += A.e.x + A.e.y;
                w_acc += A.w.x + A.w.y;
            }
#pragma unroll
            for (int o = LJ_TPP / 2; o > 0; o >>= 1) {
                fx += __shfl_xor_sync(FULL, fx, o);
                fy += __shfl_xor_sync(FULL, fy, o);
                fz += __shfl_xor_sync(FULL, fz, o);
            }
            if (act && l4 == 0) {
                b.force4[p] = make_float4(-fx, -fy, -fz, 0.f);
                if (!isfinite(fx + fy + fz)) atomicOr(&b.err[0], LJ_ERRBIT_NONFINITE);
            }
        }
        if (ENERGY) {
            // one (E_pot, W) share per warp and brick, written for every brick
            // (zeros where the warp had no particle): the warp sum in
            // double-single, stored as the (hi, lo) pair, halved exactly
            // (each pair is in two rows of a full list)
            const float2 d = warp_sum2_ds2(e_acc, w_acc);
            if ((lane & 15) == 0)
                reinterpret_cast<float2*>(b.part_f)[2 * ((size_t)bi * kBrickWarps + warp) + (lane >> 4)] =
                    make_float2(0.5f * d.x, 0.5f * d.y);
        }
        mbar_arrive1(&s_empty[buf]);   // every consumer thread: its reads of the buffer precede this
    }
}

// 1/x in FP64 for x > 0, normal: the hardware's 20-bit approximation and one
// third-order step y (1 + e + e^2), e = 1 - x y, which leaves e^3 < 2^-57.
__device__ __forceinline__ double rcp_f64(double x)
{
    double y;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    const double e = fma(-x, y, 1.0);
    return fma(y, fma(e, e, e), y);
}

// ---- 64-bit integer pair arithmetic of one species (k_force_f64) ----
// The FP64 pipe has 2 lanes per clock and SM; a 64 x 64 -> 128-bit product
// takes the integer pipes ~5 clocks per warp against 16 for one FP64
// instruction.  So the pair terms are block fixed-point numbers whose common
// exponents are set, per particle and queue drain, by the closest queued
// pair (from the FP32 scan): R = r^2 (units of 2^(sR - 2q)) is at least 2^lam
// for all of them, and
//   Y  = 2^(62 + lam) / R             t   = 1 / r^2 = Y 2^tau
//   T2 = Y^2 2^-62, T3 = T2 Y 2^-62   t^3 = T3 2^(124 + 3 tau)
//   T4 = T2^2 2^-62                   t^4 = T4 2^(186 + 4 tau)
//   g  = (T3 >> u) - Kg               t^3 - K, K = 1 / (2 sigma^6), units 2^(u + 124 + 3 tau)
//   f  = T4 |g| 2^-(63 - z)           f / c12 = t^4 (t^3 - K)
// are all below 2^62 and lose at most ~2^-57 of the closest pair's term.
// Forces and the virial are summed as 128-bit integers (no rounding at all)
// and turned into FP64 once per particle and drain.  Against exact rational
// arithmetic, errors are 2.6e-17 of S_i = sum |F_ij| at liquid densities
// (FP64 arithmetic: 1e-16).  Pairs closer than 2^-4.5 of the cutoff take the
// FP64 loop.
typedef unsigned long long u64;
typedef unsigned __int128 u128;

struct FxSums {
    __int128 x, y, z, w;   // sum f d, sum t^3 g
    u128 b;                // sum T3 >> u
};

// acc += sign * a * c, sign -1 where neg is ~0
__device__ __forceinline__ void fx_mac(__int128& acc, u64 a, u64 c, long long neg)
{
    const u128 m = (u128)(__int128)neg;
    acc += (__int128)((((u128)a * c) ^ m) - m);
}
__device__ __forceinline__ u64 fx_mul62(u64 a, u64 c) { return (u64)(((u128)a * c) >> 62); }

// Exponents of a drain, from the FP32 square r2m of its smallest distance.
struct FxScale {
    int lam, tau, u, z;
    u64 Kg;
    float ys;   // 2^(lam - 2)
    __device__ __forceinline__ bool set(const FxDev& fx, float r2m)
    {
        const float r = r2m * 0.9990234f;   // below the exact value, whatever the FP32 rounding
        const int e = (int)(__float_as_uint(r) >> 23) - 127;
        lam = e + 2 * fx.q - fx.sR;
        if (lam < 54 || lam > 62 || !(r > 1.0e-37f)) return false;
        z = (int)(7.0f * __log2f(__uint_as_float((__float_as_uint(r) & 0x007fffffu) | 0x3f800000u)));
        z = min(max(z, 0), 6);
        tau = 2 * fx.q - fx.sR - 62 - lam;
        const int xk = fx.Ke - 124 - 3 * tau;
        u = min(max(0, xk + 3), 63);
        Kg = u - xk < 64 ? fx.Km >> (u - xk) : 0ull;   // u - xk >= 3
        ys = __uint_as_float((unsigned)(lam - 2 + 127) << 23);
        return xk <= 60;
    }
};

// The pair at integer separation (dx, dy, dz).
template <bool ENERGY>
__device__ __forceinline__ bool fx_pair(const FxDev& fx, const FxScale& c, long long dx, long long dy, long long dz, FxSums& S)
{
    const long long nx = dx >> 63, ny = dy >> 63, nz = dz >> 63;
    const u64 ax = (u64)((dx ^ nx) - nx), ay = (u64)((dy ^ ny) - ny), az = (u64)((dz ^ nz) - nz);
    const u64 R = (u64)(((u128)ax * ax + (u128)ay * ay + (u128)az * az) >> fx.sR);
    if (R >= fx.Rc) return false;
    // Y: the FP32 reciprocal of R's upper word, then Y (1 + e + e^2)
    const unsigned rh = (unsigned)(R >> 32), rl = (unsigned)R;
    const unsigned y0 = (unsigned)(rcp_approx((float)rh) * c.ys);
    const int s1 = c.lam - 34;   // 20 .. 28
    const long long e = -(long long)((((u64)rh * y0) << (32 - s1)) + (((u64)rl * y0) >> s1));   // 2^64 (1 - R Y / 2^(62 + lam))
    const int eh = (int)(e >> 16);
    const long long cc = e + (((long long)eh * eh) >> 32);
    const u64 Y = ((u64)y0 << 32) + (u64)((long long)(int)(cc >> 32) * (long long)(int)y0) + __umulhi((unsigned)cc, y0);
    const u64 T2 = fx_mul62(Y, Y), T3 = fx_mul62(T2, Y), T4 = fx_mul62(T2, T2);
    const u64 T3u = T3 >> c.u;
    const long long g = (long long)(T3u - c.Kg), ng = g >> 63;
    const u64 ag = (u64)((g ^ ng) - ng);
    const u64 f = (u64)(((u128)T4 * ag) >> (63 - c.z));
    fx_mac(S.x, f, ax, ng ^ nx);
    fx_mac(S.y, f, ay, ng ^ ny);
    fx_mac(S.z, f, az, ng ^ nz);
    if (ENERGY) {
        const u128 m = (u128)(__int128)ng;
        S.w += (__int128)(((((u128)T3 * ag) >> 8) ^ m) - m);
        S.b += T3u;
    }
    return true;
}

__device__ __forceinline__ __int128 fx_shfl_add(__int128 v, int o)
{
    const u64 lo = (u64)v, hi = (u64)((u128)v >> 64);
    const u64 l2 = __shfl_xor_sync(0xffffffffu, lo, o), h2 = __shfl_xor_sync(0xffffffffu, hi, o);
    return v + (__int128)(((u128)h2 << 64) | l2);
}
// 2^n for -1022 <= n <= 1023
__device__ __forceinline__ double exp2_int(int n) { return __hiloint2double((n + 1023) << 20, 0); }
// a 2^n for normal a: the exponent bits moved or, where the result would not
// be normal, two multiplications
__device__ __forceinline__ double scale_exp2(double a, int n)
{
    const int hi = __double2hiint(a), ex = ((hi >> 20) & 0x7ff) + n;
    if (ex > 0 && ex < 2047) return __hiloint2double(hi + (n << 20), __double2loint(a));
    return a * exp2_int(n >> 1) * exp2_int(n - (n >> 1));
}
// v a 2^n
__device__ __forceinline__ double fx_to_double(__int128 v, double a, int n)
{
    return fma((double)(long long)(v >> 64), 18446744073709551616.0, (double)(u64)v) * scale_exp2(a, n);
}

// FP64 pair force (MD_PREC_FP64).  Bound: the FP64 pipe, 2 lanes per clock
// and SM (64 times fewer than FP32), where FP64 arithmetic is used, the
// integer multipliers where it is not.  TPP threads per particle scan its
// row with the FP32 offsets, four entries each and the next four in flight,
// and queue, in shared memory, the entries whose FP32 distance can lie within
// the cutoff (28 % of a row with skin 0.3 does not); the same threads then
// take the queued entries: one species in 64-bit integers (above; offsets
// from b.offx), else in FP64, the reciprocal by rcp_f64, powers of r^-2 with
// the pair constants folded, the cutoff decided on r^2's bits: 23 FP64
// instructions per pair within the cutoff with energies, against ~35 per list
// entry for a thread per particle with a division.  Work items are quarters
// of a chunk (32 particles per block), so that 4,000 particles reach 125 SMs.
// N = 256,000, energies: 1177 us -> 688 us in FP64, 307 us in integers;
// N = 4,000: a step 127 us -> 48 us in FP64, 26 us in integers.
// TPP: 4, or 16 in one-species boxes of at most an item per SM
// (BoxDev::f64_wide).
constexpr int kF64Parts = LJ_F64_WARPS;                         // work items, and (E_pot, W) shares, per chunk
constexpr int kF64Own = LJ_CHUNK / kF64Parts;                   // particles of a work item
template <bool MONO, bool ENERGY, int TPP, int RES>
__global__ void __launch_bounds__(kF64Own * TPP, RES) k_force_f64(BoxDev b)
{
    await_previous();
    constexpr int kWarps = kF64Own * TPP / 32;
    constexpr int kF64Scan = TPP == 4 ? 96 : 128;               // entries scanned between two drains of the queue
    constexpr int kF64Queue = kF64Scan + 4;                     // a particle's queue (stride 4 banks)
    __shared__ double s_ell[3][4];                     // digit (0, 1, 2) of an entry -> shift (-1, 0, 1) * edge
    __shared__ long long s_ellx[3][4];                 // the same as integers
    __shared__ uint32_t s_q[kF64Own * kF64Queue];
    __shared__ double2 s_c[LJ_MAXT * LJ_MAXT];         // 48 eps sigma^12, 24 eps sigma^6
    __shared__ double2 s_e[LJ_MAXT * LJ_MAXT];         // 4 eps sigma^12, 4 eps sigma^6
    __shared__ double s_sh[LJ_MAXT * LJ_MAXT];         // energy shift
    __shared__ unsigned long long s_rc2[LJ_MAXT * LJ_MAXT];   // rc^2 (its bits)
    __shared__ float s_near[LJ_MAXT * LJ_MAXT];        // FP32 r^2 below which an entry is queued
    __shared__ double s_red[2][kWarps];
    const LJDev* lj = b.lj;
    const int nt = b.nt;
    const int np = b.np;
    const float near1 = b.fx.near;
    const bool fxon = MONO && b.fx.on;   // integer arithmetic; the tables serve its FP64 loop's rare pairs
    for (int k = threadIdx.x; k < nt * nt; k += blockDim.x) {
        const double s2 = lj->dsig2[k], s6 = s2 * s2 * s2, e4 = lj->deps4[k];
        s_c[k] = make_double2(12.0 * e4 * s6 * s6, 6.0 * e4 * s6);
        s_e[k] = make_double2(e4 * s6 * s6, e4 * s6);
        s_sh[k] = lj->dshift[k];
        s_rc2[k] = (unsigned long long)__double_as_longlong(lj->drc2[k]);
        s_near[k] = (float)lj->drc2[k] + b.band;       // the margin of the list build's FP64 recheck
    }
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int grp = threadIdx.x / TPP, l4 = threadIdx.x % TPP;
    uint32_t* const q = s_q + grp * kF64Queue;
    const float4* posq = b.posq;
    int cur_r = -1;
    float3 ell = make_float3(0.f, 0.f, 0.f);
    for (int it = blockIdx.x; it < b.nchunk * kF64Parts; it += gridDim.x) {
        const int w = it / kF64Parts, part = it % kF64Parts;
        const int4 ch = chunk_of(b, w);
        const int r = ch.x;
        __syncthreads();   // the tables are complete; the previous item's sums are read
        if (r != cur_r) {  // block-uniform
            const RepDev& R = b.rep[r];
            // edges in the digits' units
            if (b.nrep == 1) ell = make_float3(b.ell1.x, 0.25f * b.ell1.y, 0.0625f * b.ell1.z);
            else ell = make_float3(R.ellf[0], 0.25f * R.ellf[1], 0.0625f * R.ellf[2]);
            if (threadIdx.x < 9) {
                const int c = threadIdx.x / 3, d = (int)threadIdx.x % 3 - 1;
                if (!fxon || b.nrep > 1) {
                    const double sh = (double)d * R.ell[c];
                    s_ell[c][d + 1] = sh;
                    if (MONO) s_ellx[c][d + 1] = __double2ll_rn(sh * b.fx.scale);
                } else {
                    s_ellx[c][d + 1] = (long long)d * (c == 0 ? b.fx.ell[0] : (c == 1 ? b.fx.ell[1] : b.fx.ell[2]));
                }
            }
            __syncthreads();
            cur_r = r;
        }
        if (threadIdx.x == 0 && part == 0) {
            if (w == 0) *b.any_req = 0;
            if (b.nrep == 1 ? w == 0 : w == b.rep[r].chunk_off) {
                b.disp_max[r] = 0u;
                b.rebuild_req[r] = 0;
            }
        }
        const int p = ch.y + part * kF64Own + grp;
        const bool act = p < ch.z;
        const int pa = act ? p : ch.y;
        const float4 pi = posq[pa];
        const int tb = MONO ? 0 : __float_as_int(pi.w) * nt;
        const int cnt = act ? min(b.nbr_count[p], b.K) : 0;
        long long xf = 0, yf = 0, zf = 0;
        if (fxon) {
            xf = b.offx[pa];
            yf = b.offx[np + pa];
            zf = b.offx[2 * np + pa];
        }
        bool summed = true;   // MONO: no FP64 partial sums of the four threads (their totals stand in threads 0..3)
        const uint4* row = reinterpret_cast<const uint4*>(b.nbr + (size_t)b.K * pa) + l4;
        double fx = 0.0, fy = 0.0, fz = 0.0, e = 0.0, vir = 0.0;
        int npair = 0;   // MONO: pairs within the cutoff (the shift is added once, at the end)
        // the warp's longest row bounds every lane's scans (the shuffles below are warp-wide)
        const int top = __reduce_max_sync(0xffffffffu, cnt);
        for (int s0 = 0; s0 < top; s0 += kF64Scan) {
            int nq = 0;   // queued entries of the particle (the same in its four lanes)
            float r2m = 3.0e38f;   // the smallest FP32 r^2 among them
            const int s1 = min(s0 + kF64Scan, top);
            uint4 nxt = make_uint4(0u, 0u, 0u, 0u);
            if (cnt > s0 + 4 * l4) nxt = __ldcs(row + s0 / 4);
            for (int s = s0; s < s1; s += 4 * TPP) {
                const uint4 ent = nxt;
                const int lim = cnt - (s + 4 * l4);   // entries of this thread in the block
                if (s + 4 * TPP < s1 && lim > 4 * TPP) nxt = __ldcs(row + s / 4 + TPP);   // the next block, in flight
                const uint32_t en[4] = {ent.x, ent.y, ent.z, ent.w};
                bool in[4];
                int c = 0;
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    in[u] = false;
                    if (u < lim) {
                        const float4 pj = posq[entry_slot(en[u])];
                        const float dx = fmaf(-entry_unit<0>(en[u]), ell.x, pi.x - pj.x);
                        const float dy = fmaf(-entry_unit<1>(en[u]), ell.y, pi.y - pj.y);
                        const float dz = fmaf(-entry_unit<2>(en[u]), ell.z, pi.z - pj.z);
                        const float r2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
                        in[u] = r2 < (MONO ? near1 : s_near[tb + __float_as_int(pj.w)]);
                        if (MONO && in[u]) r2m = fminf(r2m, r2);
                    }
                    c += in[u] ? 1 : 0;
                }
                int incl = c;
#pragma unroll
                for (int o = 1; o < TPP; o <<= 1) {
                    const int t = __shfl_up_sync(0xffffffffu, incl, o, TPP);
                    if (l4 >= o) incl += t;
                }
                int at = nq + incl - c;
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    if (in[u]) q[at++] = en[u];
                nq += __shfl_sync(0xffffffffu, incl, TPP - 1, TPP);
            }
            __syncwarp();
            int todo = nq;   // entries for the FP64 loop
            if (fxon) {
#pragma unroll
                for (int o = 1; o < TPP; o <<= 1) r2m = fminf(r2m, __shfl_xor_sync(0xffffffffu, r2m, o));
                FxScale c;
                FxSums S;
                S.x = S.y = S.z = S.w = 0;
                S.b = 0;
                const bool fits = nq > 0 && c.set(b.fx, r2m);
                if (fits) {
                    // the next entry's offsets are loaded while one is computed
                    long long px = 0, py = 0, pz = 0;
                    uint32_t ent = 0;
                    auto fetch = [&](int t) {
                        ent = q[t];
                        const int j = (int)entry_slot(ent);
                        px = b.offx[j];
                        py = b.offx[np + j];
                        pz = b.offx[2 * np + j];
                    };
                    if (l4 < nq) fetch(l4);
                    for (int t = l4; t < nq; t += TPP) {
                        const long long dx = (xf - px) - s_ellx[0][ent & 3u];
                        const long long dy = (yf - py) - s_ellx[1][(ent >> 2) & 3u];
                        const long long dz = (zf - pz) - s_ellx[2][(ent >> 4) & 3u];
                        if (t + TPP < nq) fetch(t + TPP);
                        if (fx_pair<ENERGY>(b.fx, c, dx, dy, dz, S) && ENERGY) ++npair;
                    }
                    todo = 0;
                }
#pragma unroll
                for (int o = 1; o < TPP; o <<= 1) {
                    S.x = fx_shfl_add(S.x, o);
                    S.y = fx_shfl_add(S.y, o);
                    S.z = fx_shfl_add(S.z, o);
                    if (ENERGY) {
                        S.w = fx_shfl_add(S.w, o);
                        S.b = (u128)fx_shfl_add((__int128)S.b, o);
                    }
                }
                if (fits) {   // thread 0, 1, 2: its component of the force; 3: the virial and the energy
                    const int g3 = c.u + 124 + 3 * c.tau;   // exponent of g
                    const __int128 v = l4 == 0 ? S.x : (l4 == 1 ? S.y : (l4 == 2 ? S.z : S.w));
                    const int n = l4 < 3 ? 63 - c.z + 186 + 4 * c.tau + g3 - b.fx.q : 8 + 124 + 3 * c.tau + g3;
                    const double d = fx_to_double(v, b.fx.c12, n);
                    fx = l4 == 0 ? fx + d : fx;
                    fy = l4 == 1 ? fy + d : fy;
                    fz = l4 == 2 ? fz + d : fz;
                    if (ENERGY && l4 == 3) {
                        vir += d;
                        e += fma(d, 1.0 / 12.0, -fx_to_double((__int128)S.b, b.fx.hb, g3));
                    }
                }
            }
            if (todo > 0) summed = false;
            double xi = 0.0, yi = 0.0, zi = 0.0, ex = 0.0, ey = 0.0, ez = 0.0;   // the FP64 loop's
            if (todo > 0) {
                xi = b.off[pa];
                yi = b.off[np + pa];
                zi = b.off[2 * np + pa];
                if (fxon && b.nrep == 1) {
                    ex = b.rep[0].ell[0];
                    ey = b.rep[0].ell[1];
                    ez = b.rep[0].ell[2];
                } else {
                    ex = s_ell[0][2];
                    ey = s_ell[1][2];
                    ez = s_ell[2][2];
                }
            }
            for (int t = l4; t < todo; t += TPP) {
                const uint32_t ent = q[t];
                const int j = (int)entry_slot(ent);
                const int gx = (int)(ent & 3u) - 1, gy = (int)((ent >> 2) & 3u) - 1, gz = (int)((ent >> 4) & 3u) - 1;
                const double dx = (xi - b.off[j]) - (gx == 0 ? 0.0 : (gx > 0 ? ex : -ex));
                const double dy = (yi - b.off[np + j]) - (gy == 0 ? 0.0 : (gy > 0 ? ey : -ey));
                const double dz = (zi - b.off[2 * np + j]) - (gz == 0 ? 0.0 : (gz > 0 ? ez : -ez));
                const double r2 = fma(dx, dx, fma(dy, dy, dz * dz));
                const int pp = MONO ? 0 : tb + b.type[j];
                // r2 < rc2 on their bits (neither is negative), not on the FP64 pipe; a NaN fails
                if ((unsigned long long)__double_as_longlong(r2) < s_rc2[pp]) {
                    const double2 c = s_c[pp];
                    const double r2i = rcp_f64(r2);
                    const double r6i = r2i * r2i * r2i;
                    const double g = r6i * fma(c.x, r6i, -c.y);   // f r^2
                    const double f = r2i * g;
                    fx = fma(f, dx, fx);
                    fy = fma(f, dy, fy);
                    fz = fma(f, dz, fz);
                    if (ENERGY) {
                        const double2 ec = s_e[pp];
                        vir += g;
                        if (MONO) {
                            e = fma(r6i, fma(ec.x, r6i, -ec.y), e);
                            ++npair;
                        } else {
                            e += fma(r6i, fma(ec.x, r6i, -ec.y), -s_sh[pp]);
                        }
                    }
                }
            }
            __syncwarp();   // the queue is read before it fills again
        }
        const bool partial = !fxon || __any_sync(0xffffffffu, !summed);   // warp-uniform
        if (partial) {
#pragma unroll
            for (int o = TPP / 2; o > 0; o >>= 1) {
                fx += __shfl_xor_sync(0xffffffffu, fx, o);
                fy += __shfl_xor_sync(0xffffffffu, fy, o);
                fz += __shfl_xor_sync(0xffffffffu, fz, o);
            }
        }
        if (act && l4 < 3) b.force64[(size_t)l4 * np + p] = l4 == 0 ? fx : (l4 == 1 ? fy : fz);
        if (act && !isfinite(fx + fy + fz)) atomicOr(&b.err[0], LJ_ERRBIT_NONFINITE);
        if (ENERGY) {
            // one (E_pot, W) share per work item
            if (partial) {
                if (MONO) e -= (double)npair * s_sh[0];
                const double de = warp_sum_d(0.5 * e), dw = warp_sum_d(0.5 * vir);
                if (lane == 0) {
                    s_red[0][warp] = de;
                    s_red[1][warp] = dw;
                }
            } else {   // every particle's sums stand in its thread 3: the energy in 2, then both summed at once
#pragma unroll
                for (int o = 1; o < TPP; o <<= 1) npair += __shfl_xor_sync(0xffffffffu, npair, o);
                const double e3 = __shfl_down_sync(0xffffffffu, e - (double)npair * s_sh[0], 1);
                double q2 = l4 == 2 ? e3 : vir;
#pragma unroll
                for (int o = TPP; o < 32; o <<= 1) q2 += __shfl_xor_sync(0xffffffffu, q2, o);
                if (lane == 2) s_red[0][warp] = 0.5 * q2;
                if (lane == 3) s_red[1][warp] = 0.5 * q2;
            }
            __syncthreads();
            if (threadIdx.x < 2) {
                double t = s_red[threadIdx.x][0];
                for (int k = 1; k < kWarps; ++k) t += s_red[threadIdx.x][k];
                b.part_f[2 * (size_t)it + threadIdx.x] = t;
            }
        }
    }
}

// ---------------------------------------------------------------------------
// All pairs (Sec. 4: the untruncated LJ interaction between all particles;
// every cutoff infinite).  With one cell per replica all offsets are from the
// box centre: d = o_i - o_j - L rint((o_i - o_j) / L) is the minimum image.
//
// FP32: a warp holds two particles and its lanes take every 32nd particle of
// the replica, so the pair arithmetic is packed over the two particles, the
// positions are staged through shared memory by the block (all loads of a
// tile in flight at once: streaming them through L1 a tile of 32 ahead waited
// for L2 at every one, 21 us at N = 2,000) and read with one load per lane and
// two pairs, and the sums meet in shuffles: no partial forces in memory and
// nothing for a last block to add up.  The minimum image
// rounds by adding and subtracting 1.5 * 2^23 (the rounding instruction runs
// at an eighth of the FP32 rate, three per pair).  Bound: issue, ~17
// instructions per pair; at N = 2,000, two warps per scheduler, latency.  Work
// items are groups of 16 particles (a block), pf_stride of them per chunk; with
// pf_stride 1 a block takes the chunk's eight groups in turn.
// N = 2,000 with energies: 21.9 us with slices of the j range per chunk,
// partial forces in memory and a last-block sum (its serial reads of 15 slices
// were half of it), 10.6 us here; N = 32,000: 1,176 -> 895 us (FP32 pipe).
// ---------------------------------------------------------------------------
constexpr int kAllWarps = 8;
constexpr int kAllThreads = 32 * kAllWarps;
constexpr int kAllGroup = 2 * kAllWarps;               // particles of a block pass
constexpr int kAllGroups = LJ_CHUNK / kAllGroup;       // passes of a chunk
constexpr int kAllTile = 2048;                         // positions staged at a time
static_assert(kAllGroups == LJ_ALL_SHARES, "one (E_pot, W) share per group");

__device__ __forceinline__ float2 dup2(float x) { return make_float2(x, x); }

template <bool MONO, bool ENERGY>
__global__ void __launch_bounds__(kAllThreads) k_force_all_f32(BoxDev b)
{
    await_previous();
    __shared__ float4 s_lj[MONO ? 1 : LJ_MAXT * LJ_MAXT];   // 4 eps sigma^12, -2 eps sigma^6, 2 eps sigma^6
    __shared__ double s_red[2][kAllWarps];
    __shared__ __align__(16) float4 s_pos[kAllTile];
    const int nt = b.nt;
    if (!MONO) {
        const LJDev* lj = b.lj;
        for (int k = threadIdx.x; k < nt * nt; k += blockDim.x)
            s_lj[k] = make_float4(lj->e12[k], -0.5f * lj->e6[k], 0.5f * lj->e6[k], 0.f);
        __syncthreads();
    }
    // one species: lengths over the power of two nearest sigma, where they are
    // staged, and the sums in units of c12 = 48 eps sigma^12 of that length (12
    // for several species, see PairSums).
    // (The list kernels' form, which needs no scale, costs an FMA with three
    // packed register operands instead of an addition: N = 32,000 836 -> 870 us.)
    const float4 one_c = b.all_1;   // 1 / length, c12, -c6 / c12, c12 / 12
    const float unit = MONO ? one_c.y : 12.f;
    const float2 nh = dup2(one_c.z);
    auto load = [&](int j) {
        float4 q = b.posq[j];
        if (MONO) {
            q.x *= one_c.x;
            q.y *= one_c.x;
            q.z *= one_c.x;
        }
        return q;
    };
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int parts = b.pf_stride;
    const float2 M = dup2(12582912.0f), nM = dup2(-12582912.0f);   // 1.5 * 2^23
    for (int it = blockIdx.x; it < b.nchunk * parts; it += gridDim.x) {
        const int w = it / parts;
        const int4 ch = chunk_of(b, w);
        const RepDev& R = b.rep[ch.x];
        if (threadIdx.x == 0 && it % parts == 0) {
            if (w == 0) *b.any_req = 0;         // the re-binning of this step has run
            if (b.nrep == 1 ? w == 0 : w == R.chunk_off) {   // clear the replica's triggers
                b.disp_max[ch.x] = 0u;
                b.rebuild_req[ch.x] = 0;
            }
        }
        // one cell: its edge is the box's (one replica: from the kernel parameters)
        float3 L = b.nrep == 1 ? b.ell1 : make_float3(R.ellf[0], R.ellf[1], R.ellf[2]);
        if (MONO) L = make_float3(L.x * one_c.x, L.y * one_c.x, L.z * one_c.x);
        const float2 ix = dup2(1.0f / L.x), iy = dup2(1.0f / L.y), iz = dup2(1.0f / L.z);
        const float2 nLx = dup2(-L.x), nLy = dup2(-L.y), nLz = dup2(-L.z);
        const int jb = b.nrep == 1 ? 0 : R.p_off, je = b.nrep == 1 ? b.n1 : R.p_off + R.n;
        double sum = 0.0;   // E_pot in the lanes below 16, W in the others
        for (int grp = it % parts; grp < kAllGroups; grp += parts) {
            const int p = ch.y + grp * kAllGroup + 2 * warp;   // the warp's particles: p and p + 1
            const bool one = p < ch.z, two = p + 1 < ch.z;     // warp-uniform
            const float4 a = load(one ? p : ch.y), c = load(two ? p + 1 : ch.y);
            const float2 nx = make_float2(-a.x, -c.x), ny = make_float2(-a.y, -c.y), nz = make_float2(-a.z, -c.z);
            const int ta = __float_as_int(a.w) * nt, tc = __float_as_int(c.w) * nt;
            float2 fx = dup2(0.f), fy = fx, fz = fx, vir = fx, eb = fx;
            // particle j against the two, masked (the particle itself, lanes past the end) by m
            auto pair = [&](const float4& q, bool masked, float2 m) {
                float2 dx = __fadd2_rn(dup2(q.x), nx), dy = __fadd2_rn(dup2(q.y), ny), dz = __fadd2_rn(dup2(q.z), nz);
                dx = __ffma2_rn(__fadd2_rn(__ffma2_rn(dx, ix, M), nM), nLx, dx);
                dy = __ffma2_rn(__fadd2_rn(__ffma2_rn(dy, iy, M), nM), nLy, dy);
                dz = __ffma2_rn(__fadd2_rn(__ffma2_rn(dz, iz, M), nM), nLz, dz);
                const float2 r2 = __ffma2_rn(dx, dx, __ffma2_rn(dy, dy, __fmul2_rn(dz, dz)));
                float2 ri = make_float2(rcp_approx(r2.x), rcp_approx(r2.y));
                if (masked) ri = make_float2(m.x != 0.f ? ri.x : 0.f, m.y != 0.f ? ri.y : 0.f);
                const float2 r6 = __fmul2_rn(__fmul2_rn(ri, ri), ri);
                float2 g;
                if (MONO) {
                    g = __fmul2_rn(r6, __fadd2_rn(r6, nh));   // f r^2, over c12
                    if (ENERGY) eb = __fadd2_rn(eb, r6);
                } else {
                    const int tj = __float_as_int(q.w);
                    const float4 u = s_lj[ta + tj], v = s_lj[tc + tj];
                    g = __fmul2_rn(r6, __ffma2_rn(make_float2(u.x, v.x), r6, make_float2(u.y, v.y)));
                    if (ENERGY) eb = __ffma2_rn(make_float2(u.z, v.z), r6, eb);
                }
                const float2 f = __fmul2_rn(ri, g);
                fx = __ffma2_rn(f, dx, fx);   // of -d: negated at the end
                fy = __ffma2_rn(f, dy, fy);
                fz = __ffma2_rn(f, dz, fz);
                if (ENERGY) vir = __fadd2_rn(vir, g);
            };
            for (int t0 = jb; t0 < je; t0 += kAllTile) {
                const int t1 = min(t0 + kAllTile, je);
                __syncthreads();   // the previous tile is no longer read
#pragma unroll
                for (int t = 0; t < kAllTile / kAllThreads; ++t) {
                    const int j = t0 + t * kAllThreads + (int)threadIdx.x;
                    if (j < t1) s_pos[j - t0] = load(j);
                }
                __syncthreads();
                if (!one) continue;
                // groups of 32: the two particles' own (both in one) and a
                // partial last one are masked, the runs between them are not
                const int full = t0 + ((t1 - t0) & ~31);
                const int own = p >= t0 && p < t1 ? t0 + ((p - t0) & ~31) : t1;
                auto run = [&](int a0, int a1) {
#pragma unroll 4
                    for (int j0 = a0; j0 < a1; j0 += 32) pair(s_pos[j0 - t0 + lane], false, dup2(1.f));
                };
                auto edge = [&](int j0) {
                    const int j = j0 + lane;
                    pair(s_pos[min(j, t1 - 1) - t0], true,
                         make_float2(j < t1 && j != p ? 1.f : 0.f, j < t1 && j != p + 1 ? 1.f : 0.f));
                };
                run(t0, min(own, full));
                if (own < t1) edge(own);
                run(own + 32, full);
                if (full < t1 && full != own) edge(full);
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                fx = __fadd2_rn(fx, make_float2(__shfl_xor_sync(0xffffffffu, fx.x, o), __shfl_xor_sync(0xffffffffu, fx.y, o)));
                fy = __fadd2_rn(fy, make_float2(__shfl_xor_sync(0xffffffffu, fy.x, o), __shfl_xor_sync(0xffffffffu, fy.y, o)));
                fz = __fadd2_rn(fz, make_float2(__shfl_xor_sync(0xffffffffu, fz.x, o), __shfl_xor_sync(0xffffffffu, fz.y, o)));
            }
            if ((lane == 0 && one) || (lane == 1 && two)) {
                const float cf = MONO ? unit * one_c.x : unit;
                const float sx = lane == 0 ? fx.x : fx.y, sy = lane == 0 ? fy.x : fy.y, sz = lane == 0 ? fz.x : fz.y;
                b.force4[p + lane] = make_float4(-cf * sx, -cf * sy, -cf * sz, 0.f);
                if (!isfinite(sx + sy + sz)) atomicOr(&b.err[0], LJ_ERRBIT_NONFINITE);
            }
            if (ENERGY) {
                // u = f r^2 / 12 - 2 eps (sigma / r)^6 (no cutoff, no shift); one species: over c12 / 12,
                // r6 (r6 + nh) + nh r6
                const float wu = vir.x + (two ? vir.y : 0.f), bu = eb.x + (two ? eb.y : 0.f);   // 0 without a first particle
                const float wv = unit * wu, ev = MONO ? one_c.w * fmaf(one_c.z, bu, wu) : wu - bu;
                const float2 d = warp_sum2_ds2(ev, wv);
                sum += (double)d.x + (double)d.y;
            }
        }
        if (ENERGY) {
            __syncthreads();   // the previous item's sums are read
            if ((lane & 15) == 0) s_red[lane >> 4][warp] = 0.5 * sum;   // each pair is seen from both ends
            __syncthreads();
            if (threadIdx.x < 2) {
                double t = 0.0;
                for (int k = 0; k < kAllWarps; ++k) t += s_red[threadIdx.x][k];
                b.part_f[2 * (size_t)it + threadIdx.x] = t;
            }
        }
    }
}

// All pairs in FP64 (MD_PREC_FP64).  Work items are (chunk of 128 particles,
// slice of the replica's particles): a block sums the chunk's forces over its
// slice into b.ap_part64, and the block that completes a chunk's last slice
// (atomic count) adds the slices in slice order (deterministic).
__device__ __forceinline__ void slice_range(const RepDev& R, int js, int nslice, int& j0, int& j1)
{
    const int len = (R.n + nslice - 1) / nslice;
    j0 = R.p_off + min(R.n, js * len);
    j1 = R.p_off + min(R.n, (js + 1) * len);
}

// The last block of chunk w: true in every thread of it.
__device__ __forceinline__ bool last_slice(const BoxDev& b, int w, int* s_flag)
{
    __syncthreads();   // this block's partials are written
    if (threadIdx.x == 0) {
        __threadfence();
        const unsigned prev = atomicAdd(&b.ap_cnt[w], 1u);
        *s_flag = prev == (unsigned)(b.ap_js - 1);
        if (*s_flag) b.ap_cnt[w] = 0u;
    }
    __syncthreads();
    const bool last = *s_flag != 0;
    if (last) __threadfence();
    return last;
}

// One thread per particle, FP64 offsets staged through shared memory; partial
// forces in b.ap_part64 (3 planes per slice).
template <bool ENERGY>
__global__ void __launch_bounds__(LJ_CHUNK) k_force_all_f64(BoxDev b)
{
    await_previous();
    constexpr int kT = 512;
    __shared__ double s_x[kT], s_y[kT], s_z[kT];
    __shared__ int s_t[kT];
    __shared__ double s_red[2][32];
    __shared__ int s_flag;
    const LJDev* lj = b.lj;
    const int nt = lj->nt;
    const int np = b.np;
    const int nitem = b.nchunk * b.ap_js;
    for (int it = blockIdx.x; it < nitem; it += gridDim.x) {
        const int w = it / b.ap_js, js = it % b.ap_js;
        const int4 ch = chunk_of(b, w);
        const RepDev& R = b.rep[ch.x];
        if (threadIdx.x == 0 && js == 0) {
            if (w == 0) *b.any_req = 0;
            if (w == R.chunk_off) {
                b.disp_max[ch.x] = 0u;
                b.rebuild_req[ch.x] = 0;
            }
        }
        const double Lx = R.L[0], Ly = R.L[1], Lz = R.L[2];
        const double ix = 1.0 / Lx, iy = 1.0 / Ly, iz = 1.0 / Lz;
        const int p = ch.y + (int)threadIdx.x;
        const bool act = p < ch.z;
        const int pa = act ? p : ch.y;
        const double xi = b.off[pa], yi = b.off[np + pa], zi = b.off[2 * np + pa];
        const int ti = b.type[pa];
        double fx = 0.0, fy = 0.0, fz = 0.0, e = 0.0, vir = 0.0;
        int j0, j1;
        slice_range(R, js, b.ap_js, j0, j1);
        for (int t0 = j0; t0 < j1; t0 += kT) {
            const int nj = min(kT, j1 - t0);
            __syncthreads();
            for (int t = threadIdx.x; t < nj; t += blockDim.x) {
                s_x[t] = b.off[t0 + t];
                s_y[t] = b.off[np + t0 + t];
                s_z[t] = b.off[2 * np + t0 + t];
                s_t[t] = b.type[t0 + t];
            }
            __syncthreads();
            if (!act) continue;
            for (int t = 0; t < nj; ++t) {
                if (t0 + t == p) continue;
                double dx = xi - s_x[t], dy = yi - s_y[t], dz = zi - s_z[t];
                dx -= Lx * rint(dx * ix);
                dy -= Ly * rint(dy * iy);
                dz -= Lz * rint(dz * iz);
                const double r2 = dx * dx + dy * dy + dz * dz;
                const int pp = ti * nt + s_t[t];
                const double r2i = 1.0 / r2;
                const double s2 = lj->dsig2[pp] * r2i;
                const double s6 = s2 * s2 * s2;
                const double f = lj->deps48[pp] * r2i * s6 * (s6 - 0.5);
                fx += f * dx;
                fy += f * dy;
                fz += f * dz;
                if (ENERGY) {
                    e += lj->deps4[pp] * s6 * (s6 - 1.0) - lj->dshift[pp];
                    vir += f * r2;
                }
            }
        }
        if (act) {
            double* part = b.ap_part64 + (size_t)js * 3 * np;
            part[p] = fx;
            part[np + p] = fy;
            part[2 * np + p] = fz;
        }
        if (ENERGY) {
            double de = 0.5 * e, dw = 0.5 * vir;
            block_sum2(de, dw, s_red);
            if (threadIdx.x == 0) {
                b.ap_pe[2 * (size_t)it] = de;
                b.ap_pe[2 * (size_t)it + 1] = dw;
            }
        }
        if (last_slice(b, w, &s_flag)) {
            for (int q = ch.y + (int)threadIdx.x; q < ch.z; q += blockDim.x) {
                double f[3] = {0.0, 0.0, 0.0};
                for (int k = 0; k < b.ap_js; ++k)
                    for (int c = 0; c < 3; ++c) f[c] += __ldcg(&b.ap_part64[(size_t)k * 3 * np + (size_t)c * np + q]);
                for (int c = 0; c < 3; ++c) b.force64[(size_t)c * np + q] = f[c];
                if (!isfinite(f[0] + f[1] + f[2])) atomicOr(&b.err[0], LJ_ERRBIT_NONFINITE);
            }
            if (ENERGY && threadIdx.x == 0) {
                double de = 0.0, dw = 0.0;
                for (int k = 0; k < b.ap_js; ++k) {
                    de += __ldcg(&b.ap_pe[2 * ((size_t)w * b.ap_js + k)]);
                    dw += __ldcg(&b.ap_pe[2 * ((size_t)w * b.ap_js + k) + 1]);
                }
                b.part_f[2 * w] = de;
                b.part_f[2 * w + 1] = dw;
            }
        }
    }
}

// A share of the FP32 forces: its (hi, lo) pair, stored where a double stands.
__device__ __forceinline__ double ds_bits_to_double(double v)
{
    return f2d(__int_as_float(__double2loint(v))) + f2d(__int_as_float(__double2hiint(v)));
}

// E_pot, E_kin, W, T per replica from the per-chunk partial sums, in a
// fixed order (deterministic): each block of LJ_THERMO_THREADS sums one item
// (a run of up to LJ_THERMO_CHUNKS chunks of one replica, pf_stride
// (E_pot, W) shares and LJ_KIN_WARPS E_kin shares per chunk).  A replica
// of one item is written out by its block directly; otherwise each block
// stores its 3 sums and the block that completes the replica's last item
// (atomic count) adds the item sums in item order and resets the count.
// Bound: the FP64 pipe of the few SMs it runs on, which it leaves idle where a
// thread has no share, and the conversions, which move bits; items of 64
// chunks instead of 256.  Beside the steps (with its fork), before / after: N =
// 4,000 11.5 / 9.9 us, 32,000 24.6 / 12.4 (there longer than the step: 20.1 ->
// 18.8 us a step), 100,000 19 / 11.8, 4M 33 / 25.
// Block `bid` of `nb`; host (nullable): the same in host memory.
__device__ __forceinline__ void thermo_items(const BoxDev& b, double* out, double* host, int with_kin, int bid, int nb)
{
    constexpr int NW = LJ_THERMO_THREADS / 32;
    static_assert(NW == 8, "a group of 8 lanes takes the warps' sums");
    __shared__ double s_red[3][NW];
    __shared__ int s_last;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // E_pot, E_kin and W over the block, in lanes 0, 8 and 16 of warp 0.  Each
    // exchange of a warp leaves half the lanes one of two sums: 6 FP64
    // additions a warp, not 15 (16 clocks of the SM's FP64 pipe each)
    auto block_sum3 = [&](double e, double w, double k) -> double {
        const bool up16 = (lane & 16) != 0, up8 = (lane & 8) != 0;
        double a = (up16 ? w : e) + __shfl_xor_sync(0xffffffffu, up16 ? e : w, 16);
        k += __shfl_xor_sync(0xffffffffu, k, 16);
        a = (up8 ? k : a) + __shfl_xor_sync(0xffffffffu, up8 ? a : k, 8);
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
        if ((lane & 7) == 0 && lane < 24) s_red[lane >> 3][warp] = a;
        __syncthreads();
        a = 0.0;
        if (warp == 0) {   // the warp sums in a fixed order
            if (lane < 24) a = s_red[lane >> 3][lane & 7];
#pragma unroll
            for (int o = 4; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
        }
        __syncthreads();
        return a;
    };
    const int which = warp == 0 && (lane & 7) == 0 && lane < 24 ? lane >> 3 : -1;   // 0 E_pot, 1 E_kin, 2 W
    auto write_out = [&](const RepDev& R, int r, double a) {
        if (which >= 0) out[4 * r + which] = a;
        if (which >= 0 && host) host[4 * r + which] = a;
        if (which == 1) out[4 * r + 3] = R.n > 1 ? 2.0 * a / (3.0 * (double)R.n - 3.0) : 0.0;
    };
    for (int it = bid; it < b.ntitem; it += nb) {
        const int4 t = b.titem[it];
        const int r = t.x;
        const RepDev& R = b.rep[r];
        double e = 0.0, w = 0.0, k = 0.0;
        const int pf = b.pf_stride;
        const double2* sh = reinterpret_cast<const double2*>(b.part_f);   // (E_pot, W) shares
        // the item's (E_pot, W) shares: those of its chunks, or, from the
        // tiled force kernel, those of its share of the replica's bricks
        int s0 = t.y * pf, s1 = t.z * pf;
        if (b.force_tiles) {
            const int q = it - R.ti_off;
            s0 = (R.brick_off + (int)(((long long)q * R.nbrick) / R.nti)) * pf;
            s1 = (R.brick_off + (int)(((long long)(q + 1) * R.nbrick) / R.nti)) * pf;
        }
        // four independent loads in flight per thread, then their sums
        const int nt4 = 4 * (int)blockDim.x;
        for (int c0 = s0; c0 < s1; c0 += nt4) {
            double2 v[4];
            const int c = c0 + (int)threadIdx.x;
#pragma unroll
            for (int u = 0; u < 4; ++u) {   // FP32 forces: (hi, lo) float pairs
                v[u] = make_double2(0.0, 0.0);
                if (c + u * LJ_THERMO_THREADS < s1) v[u] = sh[c + u * LJ_THERMO_THREADS];
            }
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (c + u * LJ_THERMO_THREADS < s1) {
                    if (b.pf_ds) {
                        e += ds_bits_to_double(v[u].x);
                        w += ds_bits_to_double(v[u].y);
                    } else {
                        e += v[u].x;
                        w += v[u].y;
                    }
                }
        }
        if (with_kin)
            for (int c0 = t.y * LJ_KIN_WARPS; c0 < t.z * LJ_KIN_WARPS; c0 += nt4) {
                double v[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int c = c0 + u * (int)blockDim.x + (int)threadIdx.x;
                    v[u] = c < t.z * LJ_KIN_WARPS ? b.part_k[c] : 0.0;
                }
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    if (c0 + u * LJ_THERMO_THREADS + (int)threadIdx.x < t.z * LJ_KIN_WARPS) k += v[u];
            }
        double a = block_sum3(e, w, k);
        if (R.nti == 1) {   // block-uniform: the replica's only item
            write_out(R, r, a);
            continue;
        }
        if (which >= 0) {
            b.part_t[3 * it + which] = a;
            __threadfence();
        }
        __syncthreads();
        if (threadIdx.x == 0) s_last = atomicAdd(&b.tcount[r], 1u) == (unsigned)(R.nti - 1);
        __syncthreads();
        if (s_last) {   // block-uniform
            __threadfence();
            e = w = k = 0.0;
            for (int i = R.ti_off + (int)threadIdx.x; i < R.ti_off + R.nti; i += blockDim.x) {
                e += __ldcg(&b.part_t[3 * i + 0]);
                k += __ldcg(&b.part_t[3 * i + 1]);
                w += __ldcg(&b.part_t[3 * i + 2]);
            }
            a = block_sum3(e, w, k);
            write_out(R, r, a);
            if (threadIdx.x == 0) b.tcount[r] = 0u;
        }
        __syncthreads();
    }
}

__global__ void __launch_bounds__(LJ_THERMO_THREADS) k_thermo(BoxDev b, double* out, int with_kin)
{
    thermo_items(b, out, nullptr, with_kin, (int)blockIdx.x, (int)gridDim.x);
}

// What follows the force kernel of a single evaluation, in one launch: blocks
// below nred reduce the energies, the others write the forces in user order
// (f nullable), and the energies and the error words go straight to pinned
// host memory.  Latency-bound: as two kernels and two copies, each waiting for
// the one before, they were a fifth of a call: N = 4,000 64.6 -> 50.1 us.
__global__ void __launch_bounds__(LJ_THERMO_THREADS) k_force_finish(BoxDev b, double* out, double* f, double* host_th,
                                                                    int* host_err, int nred)
{
    if ((int)blockIdx.x < nred) {
        if (blockIdx.x == 0 && threadIdx.x < 3) host_err[threadIdx.x] = b.err[threadIdx.x];
        thermo_items(b, out, host_th, 0, (int)blockIdx.x, nred);
        return;
    }
    constexpr int PER = LJ_THERMO_THREADS / LJ_CHUNK;   // chunks a block takes at a time
    const int np = b.np;
    for (int w = PER * ((int)blockIdx.x - nred) + (int)threadIdx.x / LJ_CHUNK; w < b.nchunk;
         w += PER * ((int)gridDim.x - nred)) {
        const int4 ch = chunk_of(b, w);
        const int p = ch.y + (int)threadIdx.x % LJ_CHUNK;
        if (p >= ch.z) continue;
        const size_t gu = (size_t)b.uid[p];
        if (b.prec == 2) {
            double q[3];
            for (int c = 0; c < 3; ++c) q[c] = b.force64[c * np + p];
            for (int c = 0; c < 3; ++c) f[3 * gu + c] = q[c];
        } else {
            const float4 q = b.force4[p];
            f[3 * gu + 0] = f2d(q.x);
            f[3 * gu + 1] = f2d(q.y);
            f[3 * gu + 2] = f2d(q.z);
        }
    }
}

}  // namespace

// The tiled force kernel's dynamic shared memory (two buffers) is above the
// default 48 KB: raise the limit once per process.
static cudaError_t tile_kernel_attrs()
{
    static cudaError_t done = cudaErrorNotReady;
    if (done == cudaErrorNotReady) {
        cudaError_t e = cudaSuccess;
        const int dm = (int)(2 * tile_buf_bytes(true)), dx = (int)(2 * tile_buf_bytes(false));
        if (e == cudaSuccess) e = cudaFuncSetAttribute(k_force_tile_f32<true, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, dm);
        if (e == cudaSuccess) e = cudaFuncSetAttribute(k_force_tile_f32<true, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, dm);
        if (e == cudaSuccess) e = cudaFuncSetAttribute(k_force_tile_f32<false, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, dx);
        if (e == cudaSuccess) e = cudaFuncSetAttribute(k_force_tile_f32<false, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, dx);
        done = e;
    }
    return done;
}

cudaError_t launch_force(const BoxDev& b, int energy, Launch l)
{
    cudaError_t e = cudaSuccess;
    if (b.all_pairs) {
        if (b.prec == 2) {
            if (energy) e = launch_kernel(k_force_all_f64<true>, l.grid, LJ_CHUNK, 0, l.s, l.early, b);
            else e = launch_kernel(k_force_all_f64<false>, l.grid, LJ_CHUNK, 0, l.s, l.early, b);
        } else if (b.nt == 1) {
            if (energy) e = launch_kernel(k_force_all_f32<true, true>, l.grid, kAllThreads, 0, l.s, l.early, b);
            else e = launch_kernel(k_force_all_f32<true, false>, l.grid, kAllThreads, 0, l.s, l.early, b);
        } else {
            if (energy) e = launch_kernel(k_force_all_f32<false, true>, l.grid, kAllThreads, 0, l.s, l.early, b);
            else e = launch_kernel(k_force_all_f32<false, false>, l.grid, kAllThreads, 0, l.s, l.early, b);
        }
        return e;
    }
    if (b.prec == 2) {
        const int wide = 16 * kF64Own, narrow = 4 * kF64Own;
        if (b.nt == 1 && b.f64_wide) {
            if (energy) e = launch_kernel(k_force_f64<true, true, 16, 1>, l.grid, wide, 0, l.s, l.early, b);
            else e = launch_kernel(k_force_f64<true, false, 16, 1>, l.grid, wide, 0, l.s, l.early, b);
        } else if (b.nt == 1) {   // 4 blocks resident: 5 and 6 (fewer registers) took 5 and 9 % longer at N = 256,000
            if (energy) e = launch_kernel(k_force_f64<true, true, 4, 4>, l.grid, narrow, 0, l.s, l.early, b);
            else e = launch_kernel(k_force_f64<true, false, 4, 4>, l.grid, narrow, 0, l.s, l.early, b);
        } else {
            if (energy) e = launch_kernel(k_force_f64<false, true, 4, 8>, l.grid, narrow, 0, l.s, l.early, b);
            else e = launch_kernel(k_force_f64<false, false, 4, 8>, l.grid, narrow, 0, l.s, l.early, b);
        }
    } else if (b.force_tiles) {
        e = tile_kernel_attrs();
        if (e != cudaSuccess) return e;
        const int th = LJ_BRICK_THREADS + 32;
        const size_t dm = 2 * tile_buf_bytes(true), dx = 2 * tile_buf_bytes(false);
        if (b.nt == 1) {
            if (energy) k_force_tile_f32<true, true><<<l.grid, th, dm, l.s>>>(b);
            else k_force_tile_f32<true, false><<<l.grid, th, dm, l.s>>>(b);
        } else {
            if (energy) k_force_tile_f32<false, true><<<l.grid, th, dx, l.s>>>(b);
            else k_force_tile_f32<false, false><<<l.grid, th, dx, l.s>>>(b);
        }
    } else if (b.force_spread) {
        const int th = LJ_SPREAD_THREADS;
        if (b.nt == 1 && b.nrep == 1) {
            if (energy) e = launch_kernel(k_force_f32<true, true, true, LJ_SPREAD_THREADS, 1>, l.grid, th, 0, l.s, l.early, b);
            else e = launch_kernel(k_force_f32<true, false, true, LJ_SPREAD_THREADS, 1>, l.grid, th, 0, l.s, l.early, b);
        } else if (b.nt == 1) {
            if (energy) e = launch_kernel(k_force_f32<true, true, false, LJ_SPREAD_THREADS, 1>, l.grid, th, 0, l.s, l.early, b);
            else e = launch_kernel(k_force_f32<true, false, false, LJ_SPREAD_THREADS, 1>, l.grid, th, 0, l.s, l.early, b);
        } else if (b.nt == 2) {
            if (energy) e = launch_kernel(k_force_f32<false, true, false, LJ_SPREAD_THREADS, 1, true>, l.grid, th, 0, l.s, l.early, b);
            else e = launch_kernel(k_force_f32<false, false, false, LJ_SPREAD_THREADS, 1, true>, l.grid, th, 0, l.s, l.early, b);
        } else {
            if (energy) e = launch_kernel(k_force_f32<false, true, false, LJ_SPREAD_THREADS, 1>, l.grid, th, 0, l.s, l.early, b);
            else e = launch_kernel(k_force_f32<false, false, false, LJ_SPREAD_THREADS, 1>, l.grid, th, 0, l.s, l.early, b);
        }
    } else if (b.nt == 1 && b.nrep == 1) {
        if (energy) e = launch_kernel(k_force_f32<true, true, true, LJ_FORCE_THREADS, 8>, l.grid, LJ_FORCE_THREADS, 0, l.s, l.early, b);
        else e = launch_kernel(k_force_f32<true, false, true, LJ_FORCE_THREADS, 8>, l.grid, LJ_FORCE_THREADS, 0, l.s, l.early, b);
    } else if (b.nt == 1) {
        if (energy) e = launch_kernel(k_force_f32<true, true, false, LJ_FORCE_THREADS, 8>, l.grid, LJ_FORCE_THREADS, 0, l.s, l.early, b);
        else e = launch_kernel(k_force_f32<true, false, false, LJ_FORCE_THREADS, 8>, l.grid, LJ_FORCE_THREADS, 0, l.s, l.early, b);
    } else if (b.nt == 2) {
        if (energy) e = launch_kernel(k_force_f32<false, true, false, LJ_FORCE_THREADS, 5, true>, l.grid, LJ_FORCE_THREADS, 0, l.s, l.early, b);
        else e = launch_kernel(k_force_f32<false, false, false, LJ_FORCE_THREADS, 6, true>, l.grid, LJ_FORCE_THREADS, 0, l.s, l.early, b);
    } else {
        if (energy) e = launch_kernel(k_force_f32<false, true, false, LJ_FORCE_THREADS, 6>, l.grid, LJ_FORCE_THREADS, 0, l.s, l.early, b);
        else e = launch_kernel(k_force_f32<false, false, false, LJ_FORCE_THREADS, 6>, l.grid, LJ_FORCE_THREADS, 0, l.s, l.early, b);
    }
    return e != cudaSuccess ? e : cudaGetLastError();
}

// Resident blocks per SM of the tiled force kernel (its persistent grid).
int force_tile_blocks_per_sm(int mono)
{
    static int occ[2] = {0, 0};
    int& o = occ[mono ? 1 : 0];
    if (o == 0 && tile_kernel_attrs() == cudaSuccess) {
        int v = 0;
        const int th = LJ_BRICK_THREADS + 32;
        cudaError_t e = mono ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(&v, k_force_tile_f32<true, true>, th,
                                                                             2 * tile_buf_bytes(true))
                             : cudaOccupancyMaxActiveBlocksPerMultiprocessor(&v, k_force_tile_f32<false, true>, th,
                                                                             2 * tile_buf_bytes(false));
        o = (e == cudaSuccess && v > 0) ? v : 2;
    }
    return o > 0 ? o : 2;
}

cudaError_t launch_force_finish(const BoxDev& b, double* out, double* f, double* host_th, int* host_err, int nred,
                                Launch l)
{
    k_force_finish<<<nred + l.grid, LJ_THERMO_THREADS, 0, l.s>>>(b, out, f, host_th, host_err, nred);
    return cudaGetLastError();
}

cudaError_t launch_thermo(const BoxDev& b, double* out, int with_kin, Launch l)
{
    k_thermo<<<l.grid, LJ_THERMO_THREADS, 0, l.s>>>(b, out, with_kin);
    return cudaGetLastError();
}
