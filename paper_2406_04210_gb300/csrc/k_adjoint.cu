// k_adjoint.cu -- reverse-mode derivative of the velocity-Verlet LJ trajectory
// and the smoothed pair-distance histogram used as a trajectory loss.
//
// The paper has no adjoint; these kernels differentiate the steps of the
// integrator (Sec. 3, Fig. 1: integrate / force / finalize; unit mass):
//   forward   vh = v_k + h/2 F(x_k); x_{k+1} = x_k + h vh; v_{k+1} = vh + h/2 F(x_{k+1})
//   reverse   lx~ = lx_{k+1} - h/2 H(x_{k+1}) lv_{k+1};  lvh = lv_{k+1} + h lx~
//             lx_k = lx~ - h/2 H(x_k) lvh;  lv_k = lvh
//   with H = Hessian of U_tot, so dF/dx = -H.  H(x_k) lvh is reused as the
//   H(x_{k+1}) lv_{k+1} term of the step before: one Hessian-vector product
//   (HVP) per step.  Parameter gradients add h/2 lv . dF/dtheta at every
//   state (twice at interior states).
// Pair HVP, with d = x_i - x_j, u_ij = u_i - u_j and the cutoff held fixed:
//   (H u)_i = sum_j [A d (d . u_ij) - f u_ij],
//   f = 48 eps s^6 (s^6 - 1/2) / r^2   (force coefficient, -phi'/r)
//   A = (phi'' - phi'/r) / r^2 = 672 eps sigma^12 / r^16 - 192 eps sigma^6 / r^10
// Parameter derivatives of F_ij = f d at fixed r and rc:
//   dF/deps = (f/eps) d,  dF/dsigma = (576 eps sigma^11 / r^14 - 144 eps sigma^5 / r^8) d
#include "ljmd_internal.cuh"

namespace {

__device__ __forceinline__ double warp_sum_d(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    return v;
}

// The tape of a replayed segment: state m's FP32 offsets in slot m, its slot ->
// user map and lists in slot idx[m] (the state at which they were last built).
struct TapeLists {
    const int* uid;
    const int* count;
    const uint32_t* nbr;
};
__device__ __forceinline__ TapeLists tape_lists(const Tape& t, int m)
{
    const char* s = t.base + (size_t)t.idx[m] * t.stride;
    return TapeLists{reinterpret_cast<const int*>(s + t.o_uid), reinterpret_cast<const int*>(s + t.o_cnt),
                     reinterpret_cast<const uint32_t*>(s + t.o_nbr)};
}
__device__ __forceinline__ const float4* tape_posq(const Tape& t, int m)
{
    return reinterpret_cast<const float4*>(t.base + (size_t)m * t.stride);
}

// State m of the replay into the tape, between the step's list update and its
// force kernel: the offsets always, the maps and lists only when this step
// built them (the box-wide rebuild word is still up) or it is the segment's
// first.  (Copied at every step the lists were 28 MB of traffic each at N =
// 32,000, behind four copy nodes per step.)
__global__ void __launch_bounds__(256) k_tape_save(BoxDev b, Tape t, int m)
{
    const bool fresh = m == 0 || *b.any_req != 0;
    char* s = t.base + (size_t)m * t.stride;
    const int i0 = blockIdx.x * blockDim.x + threadIdx.x, di = gridDim.x * blockDim.x;
    for (int i = i0; i < b.np; i += di) {
        reinterpret_cast<float4*>(s)[i] = b.posq[i];
        if (fresh) {
            reinterpret_cast<int*>(s + t.o_uid)[i] = b.uid[i];
            reinterpret_cast<int*>(s + t.o_cnt)[i] = b.nbr_count[i];
        }
    }
    if (fresh) {
        const uint4* from = reinterpret_cast<const uint4*>(b.nbr);
        uint4* to = reinterpret_cast<uint4*>(s + t.o_nbr);
        const size_t n = (size_t)b.np * (size_t)b.K / 4;
#pragma unroll 4
        for (size_t i = i0; i < n; i += di) to[i] = from[i];
    }
    if (i0 == 0) t.idx[m] = fresh ? m : t.idx[m - 1];
}

// The particles' offsets and adjoint vectors u side by side, 32 bytes each (a
// neighbour's two are one sector), u from the adjoint state (user order, FP64
// n x 3) after the half-update of this step:
//   pre = 1: lx <- lx - h/2 g;  lv <- lv + h lx;  u = lv   (then HVP of u)
//   pre = 0: u = lv                                         (first state)
__global__ void __launch_bounds__(LJ_CHUNK) k_adj_pre(BoxDev b, Tape t, int m, double* lx, double* lv, const double* g,
                                                      float4* pu, double h, int pre)
{
    const TapeLists T = tape_lists(t, m);
    const float4* posq = tape_posq(t, m);
    for (int w = blockIdx.x; w < b.nchunk; w += gridDim.x) {
        const int4 ch = chunk_of(b, w);
        const int p = ch.y + (int)threadIdx.x;
        if (p >= ch.z) continue;
        const float4 pq = posq[p];
        const size_t gu = (size_t)T.uid[p];
        double v[3], x[3], gg[3];   // every load before the stores
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            v[c] = lv[3 * gu + c];
            x[c] = pre ? lx[3 * gu + c] : 0.0;
            gg[c] = pre ? g[3 * gu + c] : 0.0;
        }
        if (pre) {
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                x[c] = x[c] - 0.5 * h * gg[c];
                v[c] = v[c] + h * x[c];
                lx[3 * gu + c] = x[c];
                lv[3 * gu + c] = v[c];
            }
        }
        pu[2 * (size_t)p] = pq;
        pu[2 * (size_t)p + 1] = make_float4((float)v[0], (float)v[1], (float)v[2], 0.f);
    }
}

// Sums of k_hvp_mono over a thread's pairs in units of c6 = 24 eps sigma^6, with
// a = -d_ij, b = u_j - u_i and q = 2 (sigma / r)^6 - 1: h = sum A (a.b) a - f b =
// -(H u)_i, and the two moments of the parameter terms, x = sum q r^-8 (u_i.a),
// y = sum r^-8 (u_i.a).
struct HvpSums {
    float hx, hy, hz;
    float2 x, y;
};

// Two pairs: separations one by one, everything from r^2 on as FP32 pairs.  In
// units of c6, with tw = 2 sigma^6: q = tw r^-6 - 1, f = r^-8 q, A = r^-10 (14 q +
// 6); the cutoff masks 1 / r^2, so a pair beyond it adds zeros.  (Units as in
// the force kernel: r^-16 alone leaves the range of FP32 with the unit of length.)
__device__ __forceinline__ void hvp_pair2(unsigned e0, const float4& q0, const float4& u0, unsigned e1,
                                          const float4& q1, const float4& u1, const float4& pi, const float4& ui,
                                          const float3& ell, float tw, float rc2, HvpSums& S)
{
    const float ax0 = fmaf(entry_unit<0>(e0), ell.x, q0.x - pi.x), ax1 = fmaf(entry_unit<0>(e1), ell.x, q1.x - pi.x);
    const float ay0 = fmaf(entry_unit<1>(e0), ell.y, q0.y - pi.y), ay1 = fmaf(entry_unit<1>(e1), ell.y, q1.y - pi.y);
    const float az0 = fmaf(entry_unit<2>(e0), ell.z, q0.z - pi.z), az1 = fmaf(entry_unit<2>(e1), ell.z, q1.z - pi.z);
    const float2 ax = make_float2(ax0, ax1), ay = make_float2(ay0, ay1), az = make_float2(az0, az1);
    const float2 bx = make_float2(u0.x - ui.x, u1.x - ui.x), by = make_float2(u0.y - ui.y, u1.y - ui.y),
                 bz = make_float2(u0.z - ui.z, u1.z - ui.z);
    const float2 r2 = __ffma2_rn(ax, ax, __ffma2_rn(ay, ay, __fmul2_rn(az, az)));
    const float2 in = make_float2(r2.x < rc2 ? 1.f : 0.f, r2.y < rc2 ? 1.f : 0.f);
    const float2 ri = __fmul2_rn(make_float2(rcp_approx(r2.x), rcp_approx(r2.y)), in);
    const float2 r6 = __fmul2_rn(__fmul2_rn(ri, ri), ri);
    const float2 r8 = __fmul2_rn(ri, r6);
    const float2 q = __ffma2_rn(make_float2(tw, tw), r6, make_float2(-1.f, -1.f));
    const float2 f = __fmul2_rn(r8, q);
    const float2 A = __fmul2_rn(__fmul2_rn(ri, r8), __ffma2_rn(make_float2(14.f, 14.f), q, make_float2(6.f, 6.f)));
    const float2 ab = __ffma2_rn(ax, bx, __ffma2_rn(ay, by, __fmul2_rn(az, bz)));
    const float2 t = __fmul2_rn(A, ab);
    const float2 nf = make_float2(-f.x, -f.y);
    const float2 hx = __ffma2_rn(t, ax, __fmul2_rn(nf, bx)), hy = __ffma2_rn(t, ay, __fmul2_rn(nf, by)),
                 hz = __ffma2_rn(t, az, __fmul2_rn(nf, bz));
    S.hx += hx.x + hx.y;
    S.hy += hy.x + hy.y;
    S.hz += hz.x + hz.y;
    const float2 ua = __ffma2_rn(make_float2(ui.x, ui.x), ax,
                                 __ffma2_rn(make_float2(ui.y, ui.y), ay, __fmul2_rn(make_float2(ui.z, ui.z), az)));
    const float2 v = __fmul2_rn(r8, ua);
    S.x = __ffma2_rn(q, v, S.x);
    S.y = __fadd2_rn(S.y, v);
}

// HVP and parameter-gradient terms at one state, one species, with the
// adjoint update that follows it:
//   g <- H u (user order, FP64);  lx <- lx - h/2 g   (when upd)
// part_g[2 q], [2 q + 1] accumulate weight * sum lam.dF/deps and lam.dF/dsigma
// over the states of the reverse sweep, q one row per warp and work item (no
// block barrier; deterministic), reduced once at its end.
// Rows, work items and threads per particle as in k_force_f32 (chunks, or 16
// particles by 64 threads in small boxes), pairs two at a time.  Bound at N =
// 32,000: the serial row's latency; 36 us with one entry in flight per thread,
// 17 us (64 registers, so that 2,000 items are one wave: 96 took 22).
template <int THREADS, int RES>
__global__ void __launch_bounds__(THREADS, RES) k_hvp_mono(BoxDev b, Tape tp, int m, const float4* __restrict__ pu,
                                                           double* lx, double* g, double h, int upd,
                                                           const double* weight, double* part_g)
{
    constexpr int PASS = THREADS / LJ_TPP;
    constexpr int PARTS = THREADS == LJ_SPREAD_THREADS ? LJ_CHUNK / PASS : 1;
    constexpr int OWN = LJ_CHUNK / PARTS;
    const TapeLists T = tape_lists(tp, m);
    const float c6 = b.c1.y, tw = b.tw_1, rc2 = b.rc2_1;
    const float inv_eps = b.lj->inv_eps[0], inv_sig = b.lj->inv_sig[0];
    const int K = b.K;
    const int grp = threadIdx.x / LJ_TPP, l4 = threadIdx.x % LJ_TPP;
    const unsigned sent = entry_make(13, b.np);
    float3 ell = make_float3(b.ell1.x, 0.25f * b.ell1.y, 0.0625f * b.ell1.z);   // edges in the digits' units
    for (int it = blockIdx.x; it < b.nchunk * PARTS; it += gridDim.x) {
        const int w = it / PARTS, part = it % PARTS;
        const int4 ch = chunk_of(b, w);
        if (b.nrep > 1) {
            const RepDev& R = b.rep[ch.x];
            ell = make_float3(R.ellf[0], 0.25f * R.ellf[1], 0.0625f * R.ellf[2]);
        }
        HvpSums S;
        S.x = S.y = make_float2(0.f, 0.f);
        const int first = ch.y + part * OWN, last = min(first + OWN, ch.z);
        for (int base = first; base < last; base += PASS) {
            const int p = base + grp;
            const bool act = p < last;
            float4 pi = make_float4(0.f, 0.f, 0.f, 0.f), ui = pi;
            int cnt = 0;
            size_t gu = 0;
            const uint4* L = reinterpret_cast<const uint4*>(T.nbr + (size_t)K * p) + l4;
            uint4 cur = make_uint4(0u, 0u, 0u, 0u);
            if (act) {
                pi = pu[2 * (size_t)p];
                ui = pu[2 * (size_t)p + 1];
                cnt = min(T.count[p], K);
                gu = 3 * (size_t)T.uid[p] + l4;
                cur = __ldcs(L);   // the row's first block (K >= 16 slots), in flight with the count
            }
            const bool out = act && l4 < 3;
            const double lx0 = out && upd ? lx[gu] : 0.0;   // this thread's component of the update
            const int nblk = (cnt + LJ_ROW_BLOCK - 1) / LJ_ROW_BLOCK;
            S.hx = S.hy = S.hz = 0.f;
            auto block4 = [&](const uint4& q) {
                const float4* n0 = pu + 2 * (size_t)entry_slot(q.x);
                const float4* n1 = pu + 2 * (size_t)entry_slot(q.y);
                const float4* n2 = pu + 2 * (size_t)entry_slot(q.z);
                const float4* n3 = pu + 2 * (size_t)entry_slot(q.w);
                const float4 p0 = __ldg(n0), v0 = __ldg(n0 + 1), p1 = __ldg(n1), v1 = __ldg(n1 + 1);
                const float4 p2 = __ldg(n2), v2 = __ldg(n2 + 1), p3 = __ldg(n3), v3 = __ldg(n3 + 1);
                hvp_pair2(q.x, p0, v0, q.y, p1, v1, pi, ui, ell, tw, rc2, S);
                hvp_pair2(q.z, p2, v2, q.w, p3, v3, pi, ui, ell, tw, rc2, S);
            };
            if (nblk > 0) {
                for (int blk = 1; blk < nblk; ++blk) {
                    const uint4 nxt = __ldcs(L + blk * LJ_TPP);   // in flight during this block
                    block4(cur);
                    cur = nxt;
                }
                const int lim = cnt - ((nblk - 1) * LJ_ROW_BLOCK + 4 * l4);   // entries past the count: the sentinel
                cur.x = lim > 0 ? cur.x : sent;
                cur.y = lim > 1 ? cur.y : sent;
                cur.z = lim > 2 ? cur.z : sent;
                cur.w = lim > 3 ? cur.w : sent;
                block4(cur);
            }
#pragma unroll
            for (int o = LJ_TPP / 2; o > 0; o >>= 1) {
                S.hx += __shfl_xor_sync(0xffffffffu, S.hx, o);
                S.hy += __shfl_xor_sync(0xffffffffu, S.hy, o);
                S.hz += __shfl_xor_sync(0xffffffffu, S.hz, o);
            }
            if (out) {
                const double hv = (double)(-c6 * (l4 == 0 ? S.hx : (l4 == 1 ? S.hy : S.hz)));
                g[gu] = hv;
                if (upd) lx[gu] = lx0 - 0.5 * h * hv;
            }
        }
        // u_i.dF/deps and u_i.dF/dsigma from the moments
        const float x = S.x.x + S.x.y, y = S.y.x + S.y.y;
        const float2 d = warp_sum2_ds2(-c6 * inv_eps * x, -6.f * c6 * inv_sig * fmaf(2.f, x, y));
        if ((threadIdx.x & 15) == 0) {
            const size_t q = (size_t)it * (THREADS / 16) + (threadIdx.x >> 4);
            part_g[q] += *weight * ((double)d.x + (double)d.y);
        }
    }
}

// The same for several species: part_g[chunk * 2P + 0..P-1] accumulates weight
// * sum lam.dF/deps and [P..2P-1] weight * sum lam.dF/dsigma per symmetric type
// pair (P = nt * nt slots; the (a, b) and (b, a) terms both land in the slot of
// min/max), summed per chunk in shared memory.
__global__ void __launch_bounds__(LJ_FORCE_THREADS) k_hvp_f32(BoxDev b, Tape tp, int m, const float4* __restrict__ pu,
                                                              double* lx, double* g, double h, int upd,
                                                              const double* weight, double* part_g)
{
    __shared__ float4 s_c[LJ_MAXT * LJ_MAXT];     // c12, c6, a12, a6
    __shared__ float4 s_g[LJ_MAXT * LJ_MAXT];     // g12, g6, 1/eps, rc2
    __shared__ float s_acc[2 * LJ_MAXT * LJ_MAXT];
    const TapeLists T = tape_lists(tp, m);
    const LJDev* lj = b.lj;
    const int nt = lj->nt;
    const int P = nt * nt;
    for (int k = threadIdx.x; k < P; k += blockDim.x) {
        s_c[k] = make_float4(lj->c12[k], lj->c6[k], lj->a12[k], lj->a6[k]);
        s_g[k] = make_float4(lj->g12[k], lj->g6[k], lj->inv_eps[k], lj->rc2[k]);
    }
    const int K = b.K;
    const int grp = threadIdx.x / LJ_TPP, l8 = threadIdx.x % LJ_TPP;
    int cur_r = -1;
    float3 ell = make_float3(0.f, 0.f, 0.f);
    for (int w = blockIdx.x; w < b.nchunk; w += gridDim.x) {
        const int4 ch = chunk_of(b, w);
        const int r = ch.x;
        if (r != cur_r) {                       // block-uniform
            const RepDev& R = b.rep[r];
            ell = make_float3(R.ellf[0], 0.25f * R.ellf[1], 0.0625f * R.ellf[2]);   // edges in the digits' units
            cur_r = r;
        }
        __syncthreads();
        for (int k = threadIdx.x; k < 2 * P; k += blockDim.x) s_acc[k] = 0.f;
        __syncthreads();
        for (int base = ch.y; base < ch.z; base += LJ_FORCE_THREADS / LJ_TPP) {
            const int p = base + grp;
            const bool act = p < ch.z;
            float4 pi = make_float4(0.f, 0.f, 0.f, 0.f), ui = pi;
            int cnt = 0;
            if (act) {
                pi = pu[2 * (size_t)p];
                ui = pu[2 * (size_t)p + 1];
                cnt = min(T.count[p], K);
            }
            const int ti = __float_as_int(pi.w);
            const uint32_t* L = T.nbr + (size_t)K * p;
            float hx = 0.f, hy = 0.f, hz = 0.f;
            for (int s = l8; s < cnt; s += LJ_TPP) {
                const unsigned ent = __ldcs(L + s);
                const size_t j = entry_slot(ent);
                const float4 pj = __ldg(pu + 2 * j);
                const float4 uj = __ldg(pu + 2 * j + 1);
                // d = (o_i - o_j) - (dx, dy, dz) * ell, one rounding per component
                const float dx = fmaf(-entry_unit<0>(ent), ell.x, pi.x - pj.x);
                const float dy = fmaf(-entry_unit<1>(ent), ell.y, pi.y - pj.y);
                const float dz = fmaf(-entry_unit<2>(ent), ell.z, pi.z - pj.z);
                const float r2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
                const int tj = __float_as_int(pj.w);
                const float4 c = s_c[ti * nt + tj], gg = s_g[ti * nt + tj];
                const bool in = r2 < gg.w;
                const float r2i = rcp_approx(r2);
                const float r6i = r2i * r2i * r2i;
                float f = r2i * r6i * fmaf(c.x, r6i, -c.y);
                float A = r2i * r2i * r6i * fmaf(c.z, r6i, -c.w);
                f = in ? f : 0.f;
                A = in ? A : 0.f;
                const float ux = ui.x - uj.x, uy = ui.y - uj.y, uz = ui.z - uj.z;
                const float du = fmaf(dx, ux, fmaf(dy, uy, dz * uz));
                const float Adu = A * du;
                hx = fmaf(Adu, dx, fmaf(-f, ux, hx));
                hy = fmaf(Adu, dy, fmaf(-f, uy, hy));
                hz = fmaf(Adu, dz, fmaf(-f, uz, hz));
                const float ld = fmaf(ui.x, dx, fmaf(ui.y, dy, ui.z * dz));
                if (in) {
                    const int q = (ti < tj ? ti : tj) * nt + (ti < tj ? tj : ti);
                    atomicAdd(&s_acc[q], f * gg.z * ld);
                    atomicAdd(&s_acc[P + q], r2i * r6i * fmaf(gg.x, r6i, -gg.y) * ld);
                }
            }
#pragma unroll
            for (int o = LJ_TPP / 2; o > 0; o >>= 1) {
                hx += __shfl_xor_sync(0xffffffffu, hx, o);
                hy += __shfl_xor_sync(0xffffffffu, hy, o);
                hz += __shfl_xor_sync(0xffffffffu, hz, o);
            }
            if (act && l8 == 0) {
                const size_t gu = (size_t)T.uid[p];
                const double hv[3] = {hx, hy, hz};
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    g[3 * gu + c] = hv[c];
                    if (upd) lx[3 * gu + c] = lx[3 * gu + c] - 0.5 * h * hv[c];
                }
            }
        }
        const double wgt = *weight;
        __syncthreads();
        for (int k = threadIdx.x; k < 2 * P; k += blockDim.x) part_g[2 * (size_t)P * w + k] += wgt * (double)s_acc[k];
    }
}

// theta_grad[q] += weight * sum over chunks of part_g[chunk * 2P + q], in a
// fixed order (one block).
__global__ void __launch_bounds__(512) k_param_reduce(const double* part_g, int nchunk, int twoP,
                                                      const double* weight, double* theta_grad)
{
    __shared__ double s_red[512 / 32];
    const double wgt = *weight;
    for (int q = 0; q < twoP; ++q) {
        double s = 0.0;
        for (int c = threadIdx.x; c < nchunk; c += blockDim.x) s += part_g[(size_t)twoP * c + q];
        s = warp_sum_d(s);
        if ((threadIdx.x & 31) == 0) s_red[threadIdx.x >> 5] = s;
        __syncthreads();
        if (threadIdx.x == 0) {
            double t = 0.0;
            for (int k = 0; k < (int)(blockDim.x >> 5); ++k) t += s_red[k];
            theta_grad[q] += wgt * t;
        }
        __syncthreads();
    }
}

// ---------------------------------------------------------------------------
// Smoothed pair-distance histogram over the current list (a trajectory
// loss):  h_k = (1/N_r) sum_{i<j, r_ij < rmax} exp(-(r_ij - c_k)^2 / (2 w^2)),
// c_k = (k + 1/2) rhist / nbins, per replica (N_r its particle count).  The
// lists must have been built at the current positions with rl >= rmax, so
// that they hold every pair below rmax.  Pairs are counted once (from the
// lower slot).  part_h[chunk * nbins + k]: per-chunk sums, reduced per replica.
//
// Bound: the special-function unit, one exponential per (pair, bin).  A warp
// takes 32 entries of a particle's row at a time, one per lane, and compacts
// the distances of the counted ones into shared memory; every 32 of them the
// lanes turn to the bins: lane l owns bins l, l + 32, ... and adds each
// distance (one broadcast load) to its own sums in registers, so a pair's
// distance is computed once for all bins and nothing is shared between lanes.
// Sums run in FP32 over 32 distances, then in double-single.  N = 32,000, 64
// bins: 1703 us with a thread per particle that walked its row once per bin,
// 61 us here.
// ---------------------------------------------------------------------------
constexpr int kHistThreads = 256;
constexpr int kHistWarps = kHistThreads / 32;

// exp(-x^2) with x scaled by sqrt(log2 e): one special-function instruction
__device__ __forceinline__ float exp2_neg_sq(float t)
{
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(-t * t));
    return y;
}

template <int NB>   // bins per lane
__global__ void __launch_bounds__(kHistThreads) k_pair_hist(BoxDev b, int nbins, float rbin, float scale, float rmax2,
                                                            double* part_h)
{
    __shared__ double s_sum[kHistWarps][32 * NB];
    __shared__ __align__(16) float s_r[kHistWarps][64];   // distances waiting for the bins: < 32 + one chunk
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u;
    float* const rr = s_r[warp];
    float ck[NB];
#pragma unroll
    for (int q = 0; q < NB; ++q) ck[q] = ((float)(lane + 32 * q) + 0.5f) * rbin;
    for (int w = blockIdx.x; w < b.nchunk; w += gridDim.x) {
        const int4 ch = chunk_of(b, w);
        const RepDev& R = b.rep[ch.x];
        const float ex = R.ellf[0], ey = 0.25f * R.ellf[1], ez = 0.0625f * R.ellf[2];   // edges in the digits' units
        float hi[NB], lo[NB];
#pragma unroll
        for (int q = 0; q < NB; ++q) hi[q] = lo[q] = 0.f;
        // 32 distances into the lane's bins
        auto batch = [&]() {
            float acc[NB];
#pragma unroll
            for (int q = 0; q < NB; ++q) acc[q] = 0.f;
#pragma unroll 2
            for (int u = 0; u < 32; u += 4) {
                const float4 r4 = *reinterpret_cast<const float4*>(rr + u);
#pragma unroll
                for (int q = 0; q < NB; ++q) {
                    acc[q] += exp2_neg_sq((r4.x - ck[q]) * scale);
                    acc[q] += exp2_neg_sq((r4.y - ck[q]) * scale);
                    acc[q] += exp2_neg_sq((r4.z - ck[q]) * scale);
                    acc[q] += exp2_neg_sq((r4.w - ck[q]) * scale);
                }
            }
#pragma unroll
            for (int q = 0; q < NB; ++q) ds_add_f(hi[q], lo[q], acc[q]);
        };
        int wait = 0;   // distances in s_r (warp-uniform)
        for (int p = ch.y + warp; p < ch.z; p += kHistWarps) {
            const float4 pi = b.posq[p];
            const int cnt = min(b.nbr_count[p], b.K);
            const uint32_t* L = b.nbr + (size_t)b.K * p;
            for (int s0 = 0; s0 < cnt; s0 += 32) {
                const int s = s0 + lane;
                bool keep = false;
                float r2 = 0.f;
                if (s < cnt) {
                    const unsigned ent = L[s];
                    const int j = (int)entry_slot(ent);
                    if (j > p) {
                        const float4 pj = b.posq[j];
                        const float dx = fmaf(-entry_unit<0>(ent), ex, pi.x - pj.x);
                        const float dy = fmaf(-entry_unit<1>(ent), ey, pi.y - pj.y);
                        const float dz = fmaf(-entry_unit<2>(ent), ez, pi.z - pj.z);
                        r2 = dx * dx + dy * dy + dz * dz;
                        keep = r2 < rmax2;
                    }
                }
                const unsigned bal = __ballot_sync(0xffffffffu, keep);
                if (keep) rr[wait + __popc(bal & lt)] = sqrtf(r2);
                wait += __popc(bal);
                __syncwarp();
                if (wait >= 32) {
                    batch();
                    const float tail = rr[32 + lane];   // the rest to the front
                    __syncwarp();
                    rr[lane] = tail;
                    wait -= 32;
                    __syncwarp();
                }
            }
        }
        if (wait > 0) {   // far points fill the last batch: their exponentials are 0
            if (lane >= wait) rr[lane] = 1.0e30f;
            __syncwarp();
            batch();
            __syncwarp();
        }
        __syncthreads();   // the previous chunk's sums are read
#pragma unroll
        for (int q = 0; q < NB; ++q) s_sum[warp][lane + 32 * q] = (double)hi[q] + (double)lo[q];
        __syncthreads();
        for (int k = threadIdx.x; k < nbins; k += kHistThreads) {
            double t = 0.0;
            for (int m = 0; m < kHistWarps; ++m) t += s_sum[m][k];
            part_h[(size_t)w * nbins + k] = t;
        }
    }
}

// per-replica histogram from the chunk sums: h[r * nbins + k] = sum / n_r.
// A block takes 32 bins of a replica, its 8 warps every eighth chunk each
// (34 us with one thread per bin over all 250 chunks of N = 32,000,
// 10 us here); the order of the sum is fixed.
__global__ void __launch_bounds__(256) k_hist_reduce(BoxDev b, int nbins, const double* part_h, double* h)
{
    __shared__ double s_red[8][32];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int nblk = (nbins + 31) / 32;
    for (int it = blockIdx.x; it < b.nrep * nblk; it += gridDim.x) {
        const int r = it / nblk, k = 32 * (it % nblk) + lane;
        const RepDev& R = b.rep[r];
        double s = 0.0;
        if (k < nbins) {
#pragma unroll 4
            for (int c = R.chunk_off + warp; c < R.chunk_off + R.nchunk; c += 8) s += part_h[(size_t)c * nbins + k];
        }
        s_red[warp][lane] = s;
        __syncthreads();
        if (warp == 0 && k < nbins) {
            for (int m = 1; m < 8; ++m) s += s_red[m][lane];
            h[(size_t)r * nbins + k] = R.n > 0 ? s / (double)R.n : 0.0;
        }
        __syncthreads();
    }
}

// gradient of sum_k coef[r, k] h_{r,k} with respect to the positions (user
// order, FP64): dh_k/dx_i = (1/N_r) sum_j g_k'(r_ij) d_ij / r_ij over i's
// full list (every pair seen from both ends), g_k' = -(r - c_k)/w^2 g_k.
// Bound by the exponentials as k_pair_hist; LJ_TPP threads per particle, as
// the force kernel, so that small boxes fill the chip (N = 32,000, 64 bins:
// 123 us with one thread per particle, 73 us here).
__global__ void __launch_bounds__(LJ_FORCE_THREADS) k_pair_hist_grad(BoxDev b, int nbins, float rbin, float scale,
                                                                     double inv_w2, float rmax2, const double* coef,
                                                                     double* grad)
{
    __shared__ float2 s_bin[256];   // c_k, -coef_k / (n w^2)
    const int grp = threadIdx.x / LJ_TPP, l4 = threadIdx.x % LJ_TPP;
    int cur_r = -1;
    float ex = 0.f, ey = 0.f, ez = 0.f;
    for (int w = blockIdx.x; w < b.nchunk; w += gridDim.x) {
        const int4 ch = chunk_of(b, w);
        if (ch.x != cur_r) {   // block-uniform
            const RepDev& R = b.rep[ch.x];
            ex = R.ellf[0];
            ey = 0.25f * R.ellf[1];   // edges in the digits' units
            ez = 0.0625f * R.ellf[2];
            __syncthreads();   // the previous replica's table is no longer read
            for (int k = threadIdx.x; k < nbins; k += blockDim.x)
                s_bin[k] = make_float2(((float)k + 0.5f) * rbin,
                                       (float)(-inv_w2 * coef[(size_t)ch.x * nbins + k] / (R.n > 0 ? (double)R.n : 1.0)));
            __syncthreads();
            cur_r = ch.x;
        }
        for (int base = ch.y; base < ch.z; base += LJ_FORCE_THREADS / LJ_TPP) {
            const int p = base + grp;
            const bool act = p < ch.z;
            const float4 pi = b.posq[act ? p : ch.y];
            const int cnt = act ? min(b.nbr_count[p], b.K) : 0;
            const uint32_t* L = b.nbr + (size_t)b.K * p;
            float gx = 0.f, gy = 0.f, gz = 0.f;
            for (int s = l4; s < cnt; s += LJ_TPP) {
                const unsigned ent = L[s];
                const float4 pj = b.posq[entry_slot(ent)];
                const float dx = fmaf(-entry_unit<0>(ent), ex, pi.x - pj.x);
                const float dy = fmaf(-entry_unit<1>(ent), ey, pi.y - pj.y);
                const float dz = fmaf(-entry_unit<2>(ent), ez, pi.z - pj.z);
                const float r2 = dx * dx + dy * dy + dz * dz;
                if (!(r2 < rmax2)) continue;
                const float r = sqrtf(r2);
                float dg = 0.f;
#pragma unroll 4
                for (int k = 0; k < nbins; ++k) {
                    const float2 c = s_bin[k];
                    const float dr = r - c.x;
                    dg = fmaf(c.y * dr, exp2_neg_sq(dr * scale), dg);
                }
                const float t = dg / r;
                gx = fmaf(t, dx, gx);
                gy = fmaf(t, dy, gy);
                gz = fmaf(t, dz, gz);
            }
#pragma unroll
            for (int o = LJ_TPP / 2; o > 0; o >>= 1) {
                gx += __shfl_xor_sync(0xffffffffu, gx, o);
                gy += __shfl_xor_sync(0xffffffffu, gy, o);
                gz += __shfl_xor_sync(0xffffffffu, gz, o);
            }
            if (act && l4 == 0) {
                const size_t gu = (size_t)b.uid[p];
                grad[3 * gu + 0] = gx;
                grad[3 * gu + 1] = gy;
                grad[3 * gu + 2] = gz;
            }
        }
    }
}

}  // namespace

cudaError_t launch_tape_save(const BoxDev& b, const Tape& t, int m, Launch l)
{
    k_tape_save<<<l.grid, 256, 0, l.s>>>(b, t, m);
    return cudaGetLastError();
}

cudaError_t launch_adj_pre(const BoxDev& b, const Tape& t, int m, double* lx, double* lv, const double* g, float4* pu,
                           double h, int pre, Launch l)
{
    k_adj_pre<<<l.grid, LJ_CHUNK, 0, l.s>>>(b, t, m, lx, lv, g, pu, h, pre);
    return cudaGetLastError();
}

cudaError_t launch_hvp(const BoxDev& b, const Tape& t, int m, const float4* pu, double* lx, double* g, double h,
                       int upd, const double* weight, double* part_g, int spread, Launch l)
{
    if (b.nt != 1)
        k_hvp_f32<<<l.grid, LJ_FORCE_THREADS, 0, l.s>>>(b, t, m, pu, lx, g, h, upd, weight, part_g);
    else if (spread)
        k_hvp_mono<LJ_SPREAD_THREADS, 16><<<l.grid, LJ_SPREAD_THREADS, 0, l.s>>>(b, t, m, pu, lx, g, h, upd, weight, part_g);
    else
        k_hvp_mono<LJ_FORCE_THREADS, 3><<<l.grid, LJ_FORCE_THREADS, 0, l.s>>>(b, t, m, pu, lx, g, h, upd, weight, part_g);
    return cudaGetLastError();
}

cudaError_t launch_param_reduce(const double* part_g, int nchunk, int twoP, const double* weight,
                                double* theta_grad, cudaStream_t s)
{
    k_param_reduce<<<1, 512, 0, s>>>(part_g, nchunk, twoP, weight, theta_grad);
    return cudaGetLastError();
}

cudaError_t launch_pair_hist(const BoxDev& b, int nbins, double rhist, double width, double rmax, double* part_h,
                             double* h, Launch l)
{
    const float rbin = (float)(rhist / nbins), rmax2 = (float)(rmax * rmax);
    // exp(-x^2 / (2 w^2)) = 2^-(scale x)^2
    const float scale = (float)sqrt(1.4426950408889634 / (2.0 * width * width));
    const int nb = (nbins + 31) / 32;   // 1 .. 8 (nbins <= 256)
    if (nb <= 1) k_pair_hist<1><<<l.grid, kHistThreads, 0, l.s>>>(b, nbins, rbin, scale, rmax2, part_h);
    else if (nb <= 2) k_pair_hist<2><<<l.grid, kHistThreads, 0, l.s>>>(b, nbins, rbin, scale, rmax2, part_h);
    else if (nb <= 4) k_pair_hist<4><<<l.grid, kHistThreads, 0, l.s>>>(b, nbins, rbin, scale, rmax2, part_h);
    else k_pair_hist<8><<<l.grid, kHistThreads, 0, l.s>>>(b, nbins, rbin, scale, rmax2, part_h);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    const int64_t items = (int64_t)b.nrep * nb;
    k_hist_reduce<<<(int)(items < 4096 ? items : 4096), 256, 0, l.s>>>(b, nbins, part_h, h);
    return cudaGetLastError();
}

cudaError_t launch_pair_hist_grad(const BoxDev& b, int nbins, double rhist, double width, double rmax,
                                  const double* coef, double* grad, Launch l)
{
    const float scale = (float)sqrt(1.4426950408889634 / (2.0 * width * width));
    k_pair_hist_grad<<<l.grid, LJ_FORCE_THREADS, 0, l.s>>>(b, nbins, (float)(rhist / nbins), scale,
                                                           1.0 / (width * width), (float)(rmax * rmax), coef, grad);
    return cudaGetLastError();
}
