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

// u (user order, FP64 n x 3) -> slot order FP32 for the HVP kernel, after
// the adjoint half-update of this step:
//   pre = 1: lx <- lx - h/2 g;  lv <- lv + h lx;  u = lv   (then HVP of u)
//   pre = 0: u = lv                                         (first state)
__global__ void __launch_bounds__(LJ_CHUNK) k_adj_pre(BoxDev b, double* lx, double* lv, const double* g,
                                                      float4* u_slot, double h, int pre)
{
    for (int w = blockIdx.x; w < b.nchunk; w += gridDim.x) {
        int4 ch = chunk_of(b, w);
        int p = ch.y + (int)threadIdx.x;
        if (p >= ch.z) continue;
        size_t gu = (size_t)b.uid[p];
        float uf[3];
        for (int c = 0; c < 3; ++c) {
            double v = lv[3 * gu + c];
            if (pre) {
                double x = lx[3 * gu + c] - 0.5 * h * g[3 * gu + c];
                lx[3 * gu + c] = x;
                v = v + h * x;
                lv[3 * gu + c] = v;
            }
            uf[c] = (float)v;
        }
        u_slot[p] = make_float4(uf[0], uf[1], uf[2], 0.f);
    }
}

// HVP and parameter-gradient terms at one state, LJ_TPP threads per particle
// (as the force kernel), with the adjoint update that follows it:
//   g <- H u (user order, FP64);  lx <- lx - h/2 g   (when upd)
// part_g[chunk * 2P + 0..P-1] accumulates weight * sum lam.dF/deps and
// [P..2P-1] weight * sum lam.dF/dsigma per symmetric type pair (P = nt * nt
// slots; the (a, b) and (b, a) terms both land in the slot of min/max) over
// the states of the reverse sweep; one reduction at its end.  MONO keeps the
// two sums in registers and accumulates one pair per warp and chunk,
// part_g[(chunk * LJ_FORCE_WARPS + warp) * 2 + 0/1], with no block barrier
// (deterministic); otherwise shared-memory atomics, one 2P row per chunk.
template <bool MONO>
__global__ void __launch_bounds__(LJ_FORCE_THREADS) k_hvp_f32(BoxDev b, const float4* __restrict__ u_slot,
                                                              double* lx, double* g, double h, int upd,
                                                              const double* weight, double* part_g)
{
    __shared__ float4 s_c[LJ_MAXT * LJ_MAXT];     // c12, c6, a12, a6
    __shared__ float4 s_g[LJ_MAXT * LJ_MAXT];     // g12, g6, 1/eps, rc2
    __shared__ float s_acc[2 * LJ_MAXT * LJ_MAXT];
    const LJDev* lj = b.lj;
    const int nt = lj->nt;
    const int P = nt * nt;
    for (int k = threadIdx.x; k < P; k += blockDim.x) {
        s_c[k] = make_float4(lj->c12[k], lj->c6[k], lj->a12[k], lj->a6[k]);
        s_g[k] = make_float4(lj->g12[k], lj->g6[k], lj->inv_eps[k], lj->rc2[k]);
    }
    __syncthreads();   // the pair tables are complete
    const float4 mc = make_float4(lj->c12[0], lj->c6[0], lj->a12[0], lj->a6[0]);
    const float4 mg = make_float4(lj->g12[0], lj->g6[0], lj->inv_eps[0], lj->rc2[0]);
    const int K = b.K;
    const int grp = threadIdx.x / LJ_TPP, l8 = threadIdx.x % LJ_TPP;
    const float4* __restrict__ posq = b.posq;
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
        if (!MONO) {   // per-chunk species-pair sums in shared memory
            __syncthreads();
            for (int k = threadIdx.x; k < 2 * P; k += blockDim.x) s_acc[k] = 0.f;
            __syncthreads();
        }
        float ge = 0.f, gs = 0.f;
        for (int base = ch.y; base < ch.z; base += LJ_FORCE_THREADS / LJ_TPP) {
            const int p = base + grp;
            const bool act = p < ch.z;
            float4 pi = make_float4(0.f, 0.f, 0.f, 0.f), ui = pi;
            int cnt = 0;
            if (act) {
                pi = posq[p];
                ui = u_slot[p];
                cnt = min(b.nbr_count[p], K);
            }
            const int ti = __float_as_int(pi.w);
            const uint32_t* L = b.nbr + (size_t)K * p;
            float hx = 0.f, hy = 0.f, hz = 0.f;
            for (int s = l8; s < cnt; s += LJ_TPP) {
                const unsigned ent = __ldcs(L + s);
                const int j = (int)entry_slot(ent);
                const float4 pj = __ldg(posq + j);
                const float4 uj = __ldg(u_slot + j);
                // d = (o_i - o_j) - (dx, dy, dz) * ell, one rounding per component
                const float dx = fmaf(-entry_unit<0>(ent), ell.x, pi.x - pj.x);
                const float dy = fmaf(-entry_unit<1>(ent), ell.y, pi.y - pj.y);
                const float dz = fmaf(-entry_unit<2>(ent), ell.z, pi.z - pj.z);
                const float r2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
                float4 c, gg;
                int pp = 0;
                if (MONO) {
                    c = mc;
                    gg = mg;
                } else {
                    pp = ti * nt + __float_as_int(pj.w);
                    c = s_c[pp];
                    gg = s_g[pp];
                }
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
                const float dsg = in ? r2i * r6i * fmaf(gg.x, r6i, -gg.y) * ld : 0.f;
                const float dep = f * gg.z * ld;
                if (MONO) {
                    ge += dep;
                    gs += dsg;
                } else if (in) {
                    const int a = ti, bb = __float_as_int(pj.w);
                    const int q = (a < bb ? a : bb) * nt + (a < bb ? bb : a);
                    atomicAdd(&s_acc[q], dep);
                    atomicAdd(&s_acc[P + q], dsg);
                }
            }
#pragma unroll
            for (int o = LJ_TPP / 2; o > 0; o >>= 1) {
                hx += __shfl_xor_sync(0xffffffffu, hx, o);
                hy += __shfl_xor_sync(0xffffffffu, hy, o);
                hz += __shfl_xor_sync(0xffffffffu, hz, o);
            }
            if (act && l8 == 0) {
                const size_t gu = (size_t)b.uid[p];
                const double hv[3] = {hx, hy, hz};
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    g[3 * gu + c] = hv[c];
                    if (upd) lx[3 * gu + c] = lx[3 * gu + c] - 0.5 * h * hv[c];
                }
            }
        }
        const double wgt = *weight;
        if (MONO) {
            // one (d/deps, d/dsigma) share per warp and chunk (no block barrier)
            const double de = warp_sum_ds(ge), ds = warp_sum_ds(gs);   // double-single warp sums
            if ((threadIdx.x & 31) == 0) {
                const size_t q = (size_t)w * LJ_FORCE_WARPS + (threadIdx.x >> 5);
                part_g[2 * q] += wgt * de;
                part_g[2 * q + 1] += wgt * ds;
            }
        } else {
            __syncthreads();
            for (int k = threadIdx.x; k < 2 * P; k += blockDim.x)
                part_g[2 * (size_t)P * w + k] += wgt * (double)s_acc[k];
        }
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

cudaError_t launch_adj_pre(const BoxDev& b, double* lx, double* lv, const double* g, float4* u_slot, double h,
                           int pre, Launch l)
{
    k_adj_pre<<<l.grid, LJ_CHUNK, 0, l.s>>>(b, lx, lv, g, u_slot, h, pre);
    return cudaGetLastError();
}

cudaError_t launch_hvp(const BoxDev& b, const float4* u_slot, double* lx, double* g, double h, int upd,
                       const double* weight, double* part_g, Launch l)
{
    if (b.nt == 1) k_hvp_f32<true><<<l.grid, LJ_FORCE_THREADS, 0, l.s>>>(b, u_slot, lx, g, h, upd, weight, part_g);
    else k_hvp_f32<false><<<l.grid, LJ_FORCE_THREADS, 0, l.s>>>(b, u_slot, lx, g, h, upd, weight, part_g);
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
