// k_integrate.cu -- velocity-Verlet half steps and state transfer kernels.
//
// Sec. 3 (Code structure, Fig. 1): the integrator module's `integrate`
// (half kick + drift) and `finalize` (half kick) slots run around the force
// evaluation.  The finalize of step s and the integrate of step s+1 touch the
// same particle data back to back, so LJ_STEP_MID fuses them into one pass
// (the arithmetic is unchanged: two separate half kicks, same roundings).
//
// Accumulation type ACC: 0 = double-single (two FP32 words; HAL's MD "mixed
// precision", Sec. 3), 1 = FP64.  FORCE64 selects FP64 forces.
// Per particle and step the kernel also measures the displacement since the
// last list build (FP32, from the cell-relative copies) and raises the
// replica's rebuild trigger when it exceeds skin/2 (Sec. 5: rebuilds become
// more frequent at higher temperature).
#include "ljmd_internal.cuh"

namespace {

__device__ __forceinline__ double warp_sum_d(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    return v;
}

// Andersen-like collision of particle u of replica r after the finalize of
// step `step` (see md_set_thermostat): true and the new velocity in g when word 0 of
// philox((u, step lo, step hi, 0), seed + replica) is below
// the threshold; Gaussians by Box-Muller.  All lanes of the warp call it (act:
// the lane has a particle).  The FP64 logarithm and the sine pair are long
// dependent chains on a slow pipe, and few lanes collide in a step: up to
// kFewHits of them are taken in turn by the whole warp, even lanes computing
// the first Box-Muller pair and odd lanes the second at the same time.
constexpr int kFewHits = 2;
__device__ __forceinline__ void box_muller(unsigned w0, unsigned w1, double& rs, double& rc)
{
    const double inv32 = 1.0 / 4294967296.0;
    const double r = sqrt(-2.0 * log(((double)w0 + 0.5) * inv32));
    double s, c;
    sincospi(2.0 * (((double)w1 + 0.5) * inv32), &s, &c);
    rs = r * s;
    rc = r * c;
}
__device__ __forceinline__ bool tstat_collide(const BoxDev& b, const RepDev& R, int r, unsigned u, bool act,
                                              long long step, double g[3])
{
    const unsigned long long key = b.tstat_seed + (unsigned long long)r;
    const uint2 k = make_uint2((unsigned)key, (unsigned)(key >> 32));
    const unsigned slo = (unsigned)step, shi = (unsigned)((unsigned long long)step >> 32);
    const uint4 x = philox4x32_10(make_uint4(u, slo, shi, 0u), k);
    const bool hit = act && x.x < b.tstat_thr;
    unsigned todo = __ballot_sync(0xffffffffu, hit);
    if (todo == 0u) return false;   // warp-uniform
    uint4 y = make_uint4(0u, 0u, 0u, 0u);
    if (hit) y = philox4x32_10(make_uint4(u, slo, shi, 1u), k);
    const double sd = sqrt(b.tstat_T[r]);
    double rs, rc;
    if (__popc(todo) <= kFewHits) {
        const bool odd = (threadIdx.x & 1) != 0;
        for (; todo; todo &= todo - 1u) {
            const int src = __ffs(todo) - 1;
            const unsigned a0 = __shfl_sync(0xffffffffu, x.y, src), a1 = __shfl_sync(0xffffffffu, x.z, src);
            const unsigned b0 = __shfl_sync(0xffffffffu, y.x, src), b1 = __shfl_sync(0xffffffffu, y.y, src);
            box_muller(odd ? b0 : a0, odd ? b1 : a1, rs, rc);
            const double g0 = __shfl_sync(0xffffffffu, rc, 0), g1 = __shfl_sync(0xffffffffu, rs, 0);
            const double g2 = __shfl_sync(0xffffffffu, rc, 1);
            if ((int)(threadIdx.x & 31) == src) {
                g[0] = sd * g0;
                g[1] = sd * g1;
                g[2] = sd * g2;
            }
        }
    } else if (hit) {
        box_muller(x.y, x.z, rs, rc);
        g[0] = sd * rc;
        g[1] = sd * rs;
        box_muller(y.x, y.y, rs, rc);
        g[2] = sd * rc;
    }
    return hit;
}

// The collisions of a graph's steps, drawn at its head: the FP64 chain above
// would otherwise stand in every step's integrator (5.6 of 14.3 us at N =
// 2,000), while here all steps and particles draw at once.
__global__ void __launch_bounds__(LJ_CHUNK) k_tstat_draw(BoxDev b, int nsteps, unsigned* hit_bits, double* gs)
{
    for (int it = blockIdx.x; it < nsteps * b.nchunk; it += gridDim.x) {
        const int step = it / b.nchunk, w = it % b.nchunk;
        const int4 ch = chunk_of(b, w);
        const RepDev& R = b.rep[ch.x];
        const int q = ch.y + (int)threadIdx.x;   // slot before any sort
        double g[3] = {0.0, 0.0, 0.0};
        const bool hit = tstat_collide(b, R, ch.x, (unsigned)(q - R.p_off), q < ch.z, *b.step_ctr + step, g);
        const unsigned bits = __ballot_sync(0xffffffffu, hit);
        if ((threadIdx.x & 31) == 0 && q < ch.z) hit_bits[(size_t)step * (b.np / 32) + q / 32] = bits;
        if (hit)
            for (int c = 0; c < 3; ++c) gs[((size_t)step * b.np + q) * 3 + c] = g[c];
    }
}
// the same, read back by the integrator
__device__ __forceinline__ bool tstat_drawn(const BoxDev& b, const RepDev& R, int uid, int sidx, double g[3])
{
    const int q = b.nrep == 1 ? uid : R.p_off + (uid - R.u_off);
    if (!((b.tstat_hit[(size_t)sidx * (b.np / 32) + q / 32] >> (q & 31)) & 1u)) return false;
    for (int c = 0; c < 3; ++c) g[c] = b.tstat_g[((size_t)sidx * b.np + q) * 3 + c];
    return true;
}

// The all-pairs form (one cell per replica, offsets from the box centre):
// the drift keeps each offset in [-L/2, L/2) itself, counting the image, so
// the form needs no re-binning between steps (there are no lists).
__device__ __forceinline__ void wrap_ds(const BoxDev& b, const RepDev& R, int c, int p, float& oh, float& ol)
{
    const float lh = (float)R.L[c], ll = (float)(R.L[c] - (double)lh);
    if (oh >= 0.5f * lh) {
        ds_add_ds(oh, ol, -lh, -ll);
        b.img[c * b.np + p] += 1;
    } else if (oh < -0.5f * lh) {
        ds_add_ds(oh, ol, lh, ll);
        b.img[c * b.np + p] -= 1;
    }
}
__device__ __forceinline__ void wrap_d(const BoxDev& b, const RepDev& R, int c, int p, double& x)
{
    if (x >= 0.5 * R.L[c]) {
        x -= R.L[c];
        b.img[c * b.np + p] += 1;
    } else if (x < -0.5 * R.L[c]) {
        x += R.L[c];
        b.img[c * b.np + p] -= 1;
    }
}

// sidx: this launch finalizes step (*b.step_ctr + sidx) (MID and LAST modes).
// Bound by HBM (~148 B per particle); all loads are issued before the stores:
// 105 -> 98 us a step at 4M particles.
template <int ACC, bool FORCE64, int MODE, bool ENERGY, bool TSTAT>
__global__ void __launch_bounds__(LJ_CHUNK) k_integrate(BoxDev b, double dt, int sidx,
                                                        cudaGraphConditionalHandle cond)
{
    await_previous();
    const int np = b.np;
    const double hdt = 0.5 * dt;
    float dt_h, dt_l;
    ds_from_double(dt, dt_h, dt_l);
    const float hdt_f = (float)hdt;
    float* offf = reinterpret_cast<float*>(b.off);
    float* velf = reinterpret_cast<float*>(b.vel);
    for (int w = blockIdx.x; w < b.nchunk; w += gridDim.x) {
        int4 ch = chunk_of(b, w);
        int r = ch.x;
        int p = ch.y + (int)threadIdx.x;
        double ek = 0.0;
        float ekf = 0.f;   // double-single state: FP32 per particle
        unsigned dmax = 0u;
        // thermostat collision after the finalize of this step
        double g[3] = {0.0, 0.0, 0.0};
        bool hit = false;
        if (TSTAT && MODE != LJ_STEP_FIRST) {
            const RepDev& R = b.rep[r];
            const int uid = p < ch.z ? b.uid[p] : 0;
            if (b.tstat_hit) hit = p < ch.z && tstat_drawn(b, R, uid, sidx, g);
            else hit = tstat_collide(b, R, r, (unsigned)(uid - R.u_off), p < ch.z, *b.step_ctr + sidx, g);
        }
        if (p < ch.z) {
            // every load before the stores (the arrays may alias as far as
            // the compiler knows: a load behind a store waits its turn)
            float vh3[3], vl3[3], oh3[3], ol3[3];
            double vd3[3], od3[3];
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                if (ACC == 0) {
                    vh3[c] = velf[c * np + p];
                    vl3[c] = velf[3 * np + c * np + p];
                    if (MODE != LJ_STEP_LAST) {
                        oh3[c] = offf[c * np + p];
                        ol3[c] = offf[3 * np + c * np + p];
                    }
                } else {
                    vd3[c] = b.vel[c * np + p];
                    if (MODE != LJ_STEP_LAST) od3[c] = b.off[c * np + p];
                }
            }
            const bool drift = MODE != LJ_STEP_LAST;
            const int type = drift ? b.type[p] : 0;
            const float4 rf = drift && !b.all_pairs ? b.ref[p] : make_float4(0.f, 0.f, 0.f, 0.f);
            double F[3];
            if (FORCE64) {
                F[0] = b.force64[p];
                F[1] = b.force64[np + p];
                F[2] = b.force64[2 * np + p];
            } else {
                float4 f4 = b.force4[p];
                F[0] = f4.x;
                F[1] = f4.y;
                F[2] = f4.z;
            }
            float o[3];
            if (ACC == 0) {
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    float vh = vh3[c], vl = vl3[c];
                    float inc = hdt_f * (float)F[c];
                    if (MODE != LJ_STEP_FIRST) {
                        ds_add_f(vh, vl, inc);
                        if (hit) ds_from_double(g[c], vh, vl);
                        if (ENERGY) ekf += vh * vh;
                    }
                    if (MODE != LJ_STEP_LAST) {
                        ds_add_f(vh, vl, inc);
                        float oh = oh3[c], ol = ol3[c];
                        float ph, pl;
                        ds_mul_ds(dt_h, dt_l, vh, vl, ph, pl);
                        ds_add_ds(oh, ol, ph, pl);
                        if (b.all_pairs) wrap_ds(b, b.rep[r], c, p, oh, ol);
                        offf[c * np + p] = oh;
                        offf[3 * np + c * np + p] = ol;
                        o[c] = oh;
                    }
                    velf[c * np + p] = vh;
                    velf[3 * np + c * np + p] = vl;
                }
            } else {
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    double v = vd3[c];
                    if (MODE != LJ_STEP_FIRST) {
                        v = v + hdt * F[c];
                        if (hit) v = g[c];
                        if (ENERGY) ek += v * v;
                    }
                    if (MODE != LJ_STEP_LAST) {
                        v = v + hdt * F[c];
                        double x = od3[c] + dt * v;
                        if (b.all_pairs) wrap_d(b, b.rep[r], c, p, x);
                        b.off[c * np + p] = x;
                        if (FORCE64 && b.offx) b.offx[c * np + p] = __double2ll_rn(x * b.fx.scale);
                        o[c] = __double2float_rn(x);
                    }
                    b.vel[c * np + p] = v;
                }
            }
            if (MODE != LJ_STEP_LAST && b.all_pairs) {
                b.posq[p] = make_float4(o[0], o[1], o[2], __int_as_float(type));
            } else if (MODE != LJ_STEP_LAST) {
                b.posq[p] = make_float4(o[0], o[1], o[2], __int_as_float(type));
                float ddx = o[0] - rf.x, ddy = o[1] - rf.y, ddz = o[2] - rf.z;
                float d2 = ddx * ddx + ddy * ddy + ddz * ddz;
                if (!(d2 <= 3.0e38f)) d2 = 3.0e38f;   // NaN or inf: force a rebuild
                dmax = __float_as_uint(d2);
            }
        }
        if (MODE != LJ_STEP_LAST) {
            unsigned m = __reduce_max_sync(0xffffffffu, dmax);
            if ((threadIdx.x & 31) == 0 && __uint_as_float(m) > b.disp_thr2) {
                atomicMax(&b.disp_max[r], m);
                atomicOr(b.any_req, 1);
                if (cond) cudaGraphSetConditional(cond, 1u);
            }
        }
        if (ENERGY && MODE != LJ_STEP_FIRST) {
            // one E_kin share per warp and chunk (no block barrier); the
            // double-single state sums its FP32 squares in double-single
            const double s = ACC == 0 ? 0.5 * warp_sum_ds(ekf) : warp_sum_d(0.5 * ek);
            if ((threadIdx.x & 31) == 0) b.part_k[(size_t)w * LJ_KIN_WARPS + (threadIdx.x >> 5)] = s;
        }
    }
}

template <int ACC, bool FORCE64>
cudaError_t launch_integrate_t(const BoxDev& b, int mode, int energy, double dt, int sidx,
                               cudaGraphConditionalHandle cond, Launch l)
{
#define LJ_INT_CASE(M, E)                                                                       \
    do {                                                                                        \
        return launch_kernel(b.tstat_thr ? k_integrate<ACC, FORCE64, M, E, true> : k_integrate<ACC, FORCE64, M, E, false>, \
                             l.grid, LJ_CHUNK, 0, l.s, l.early, b, dt, sidx, cond);                     \
    } while (0)
    if (mode == LJ_STEP_FIRST) LJ_INT_CASE(LJ_STEP_FIRST, false);
    else if (mode == LJ_STEP_MID) {
        if (energy) LJ_INT_CASE(LJ_STEP_MID, true);
        else LJ_INT_CASE(LJ_STEP_MID, false);
    } else {
        if (energy) LJ_INT_CASE(LJ_STEP_LAST, true);
        else LJ_INT_CASE(LJ_STEP_LAST, false);
    }
#undef LJ_INT_CASE
}

// ---------------------------------------------------------------------------
// State transfer.  User-order arrays (n x 3 FP64 AoS, device memory) <->
// the box's slot arrays.  Before the first build, slot p of replica r holds
// user particle u_off + (p - p_off).
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(LJ_CHUNK) k_upload(BoxDev b, const double* pos,
                                                     const double* vel, const int* type,
                                                     int set_vel)
{
    const int np = b.np;
    for (int w = blockIdx.x; w < b.nchunk; w += gridDim.x) {
        int4 ch = chunk_of(b, w);
        int p = ch.y + (int)threadIdx.x;
        if (p >= ch.z) continue;
        const RepDev& R = b.rep[ch.x];
        int gu = R.u_off + (p - R.p_off);
        double x3[3], v3[3];   // every load before the stores
        const int ty = type ? type[gu] : 0;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            x3[c] = pos[3 * (size_t)gu + c];
            v3[c] = set_vel && vel ? vel[3 * (size_t)gu + c] : 0.0;
        }
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            double x = x3[c];
            double L = R.L[c];
            double f = floor_div(x, R.wrap_hi[c], L);
            b.xabs[c * np + p] = x - L * f;
            b.img[c * np + p] = (int)f;
            if (set_vel) {
                const double v = v3[c];
                if (b.prec == 0) {
                    float h, lo;
                    ds_from_double(v, h, lo);
                    float* vf = reinterpret_cast<float*>(b.vel);
                    vf[c * np + p] = h;
                    vf[3 * np + c * np + p] = lo;
                } else {
                    b.vel[c * np + p] = v;
                }
            }
        }
        b.uid[p] = gu;
        if (type) b.type[p] = ty;
    }
}

// Current positions (wrapped into [0, L), image counts adjusted), velocities.
// At 4M particles 479 us with an FP64 division and four FP32-to-FP64
// conversions per component, 235 us without and with the loads together
// (k_upload 387 -> 129 us).
__global__ void __launch_bounds__(LJ_CHUNK) k_download(BoxDev b, double* pos, double* vel,
                                                       int* img)
{
    const int np = b.np;
    for (int w = blockIdx.x; w < b.nchunk; w += gridDim.x) {
        int4 ch = chunk_of(b, w);
        int p = ch.y + (int)threadIdx.x;
        if (p >= ch.z) continue;
        const RepDev& R = b.rep[ch.x];
        const int gu = b.uid[p];
        const int local = b.cell[p] - R.cell_off;
        const float* of = reinterpret_cast<const float*>(b.off);
        const float* vf = reinterpret_cast<const float*>(b.vel);
        float fo[6], fv[6];
        double o[3], v[3];
        int im3[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) {   // every load before the stores
            im3[c] = b.img[c * np + p];
            if (b.prec == 0) {
                fo[c] = of[c * np + p];
                fo[3 + c] = of[3 * np + c * np + p];
                fv[c] = vf[c * np + p];
                fv[3 + c] = vf[3 * np + c * np + p];
            } else {
                o[c] = b.off[c * np + p];
                v[c] = b.vel[c * np + p];
            }
        }
        int cc[3];
        cc[0] = local % R.nc[0];
        cc[1] = (local / R.nc[0]) % R.nc[1];
        cc[2] = local / (R.nc[0] * R.nc[1]);
        if (b.prec == 0) {
            ds_to_double3(fo, fo + 3, o);
            ds_to_double3(fv, fv + 3, v);
        }
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            double x = fma(half_above(cc[c]), R.ell[c], o[c]);
            int im = im3[c];
            const double L = R.L[c];
            const double f = floor_div(x, R.wrap_hi[c], L);
            if (f != 0.0) {
                x = x - L * f;
                im += (int)f;
            }
            if (pos) pos[3 * (size_t)gu + c] = x;
            if (vel) vel[3 * (size_t)gu + c] = v[c];
            if (img) img[3 * (size_t)gu + c] = im;
        }
    }
}

__global__ void __launch_bounds__(LJ_CHUNK) k_force_out(BoxDev b, double* f)
{
    const int np = b.np;
    for (int w = blockIdx.x; w < b.nchunk; w += gridDim.x) {
        int4 ch = chunk_of(b, w);
        int p = ch.y + (int)threadIdx.x;
        if (p >= ch.z) continue;
        size_t gu = (size_t)b.uid[p];
        if (b.prec == 2) {
            for (int c = 0; c < 3; ++c) f[3 * gu + c] = b.force64[c * np + p];
        } else {
            float4 q = b.force4[p];
            f[3 * gu + 0] = q.x;
            f[3 * gu + 1] = q.y;
            f[3 * gu + 2] = q.z;
        }
    }
}

__global__ void __launch_bounds__(LJ_CHUNK) k_get_nlist(BoxDev b, int* count, long long* nbr,
                                                        long long cap, double* pos)
{
    const int np = b.np;
    for (int w = blockIdx.x; w < b.nchunk; w += gridDim.x) {
        int4 ch = chunk_of(b, w);
        int p = ch.y + (int)threadIdx.x;
        if (p >= ch.z) continue;
        long long gu = b.uid[p];
        int cnt = b.nbr_count[p];
        count[gu] = cnt;
        if (pos)
            for (int c = 0; c < 3; ++c) pos[3 * gu + c] = b.xabs[c * np + p];
        if (nbr) {
            int m = cnt < b.K ? cnt : b.K;
            if ((long long)m > cap) m = (int)cap;
            const uint32_t* lp = b.nbr + (size_t)b.K * p;
            for (int s = 0; s < m; ++s) nbr[gu * cap + s] = b.uid[entry_slot(lp[s])];
        }
    }
}

}  // namespace

cudaError_t launch_integrate(const BoxDev& b, int mode, int energy, double dt, int sidx,
                             cudaGraphConditionalHandle cond, Launch l)
{
    if (b.prec == 0) return launch_integrate_t<0, false>(b, mode, energy, dt, sidx, cond, l);
    if (b.prec == 1) return launch_integrate_t<1, false>(b, mode, energy, dt, sidx, cond, l);
    return launch_integrate_t<1, true>(b, mode, energy, dt, sidx, cond, l);
}

namespace {
__global__ void k_step_advance(long long* ctr, long long n)
{
    if (blockIdx.x == 0 && threadIdx.x == 0) *ctr += n;
}
}  // namespace

cudaError_t launch_tstat_draw(const BoxDev& b, int nsteps, unsigned* hit, double* g, Launch l)
{
    k_tstat_draw<<<l.grid, LJ_CHUNK, 0, l.s>>>(b, nsteps, hit, g);
    return cudaGetLastError();
}

cudaError_t launch_step_advance(long long* ctr, long long n, cudaStream_t s)
{
    k_step_advance<<<1, 32, 0, s>>>(ctr, n);
    return cudaGetLastError();
}

cudaError_t launch_upload(const BoxDev& b, const double* pos, const double* vel, const int* type,
                          int set_vel, Launch l)
{
    k_upload<<<l.grid, LJ_CHUNK, 0, l.s>>>(b, pos, vel, type, set_vel);
    return cudaGetLastError();
}

cudaError_t launch_download(const BoxDev& b, double* pos, double* vel, int* img, Launch l)
{
    k_download<<<l.grid, LJ_CHUNK, 0, l.s>>>(b, pos, vel, img);
    return cudaGetLastError();
}

cudaError_t launch_force_out(const BoxDev& b, double* f, Launch l)
{
    k_force_out<<<l.grid, LJ_CHUNK, 0, l.s>>>(b, f);
    return cudaGetLastError();
}

cudaError_t launch_get_nlist(const BoxDev& b, int* count, long long* nbr, long long cap,
                             double* pos, Launch l)
{
    k_get_nlist<<<l.grid, LJ_CHUNK, 0, l.s>>>(b, count, nbr, cap, pos);
    return cudaGetLastError();
}

namespace {
// Positions from (cell, offset) into xabs/img in place (wrapped), before the
// cell grid is changed.
__global__ void __launch_bounds__(LJ_CHUNK) k_materialize(BoxDev b)
{
    const int np = b.np;
    for (int w = blockIdx.x; w < b.nchunk; w += gridDim.x) {
        int4 ch = chunk_of(b, w);
        int p = ch.y + (int)threadIdx.x;
        if (p >= ch.z) continue;
        const RepDev& R = b.rep[ch.x];
        int local = b.cell[p] - R.cell_off;
        int cc[3];
        cc[0] = local % R.nc[0];
        cc[1] = (local / R.nc[0]) % R.nc[1];
        cc[2] = local / (R.nc[0] * R.nc[1]);
        for (int c = 0; c < 3; ++c) {
            double o;
            if (b.prec == 0) {
                const float* of = reinterpret_cast<const float*>(b.off);
                o = (double)of[c * np + p] + (double)of[3 * np + c * np + p];
            } else {
                o = b.off[c * np + p];
            }
            double x = ((double)cc[c] + 0.5) * R.ell[c] + o;
            double L = R.L[c];
            double f = floor(x / L);
            int im = b.img[c * np + p];
            if (f != 0.0) {
                x = x - L * f;
                im += (int)f;
            }
            b.xabs[c * np + p] = x;
            b.img[c * np + p] = im;
        }
    }
}
}  // namespace

namespace {
__global__ void __launch_bounds__(LJ_CHUNK) k_fix(BoxDev b)
{
    for (int w = blockIdx.x; w < b.nchunk; w += gridDim.x) {
        const int4 ch = chunk_of(b, w);
        const int p = ch.y + (int)threadIdx.x;
        if (p >= ch.z) continue;
        for (int c = 0; c < 3; ++c) b.offx[c * b.np + p] = __double2ll_rn(b.off[c * b.np + p] * b.fx.scale);
    }
}
}  // namespace

cudaError_t launch_fix(const BoxDev& b, Launch l)
{
    k_fix<<<l.grid, LJ_CHUNK, 0, l.s>>>(b);
    return cudaGetLastError();
}

cudaError_t launch_materialize(const BoxDev& b, Launch l)
{
    k_materialize<<<l.grid, LJ_CHUNK, 0, l.s>>>(b);
    return cudaGetLastError();
}
