// nd_field_impl.cuh -- field evaluation and time stepping kernels (templates;
// instantiated by nd_fused_f32.cu, nd_fused_f64.cu, nd_glob_f32.cu, nd_glob_f64.cu).
//
// Two drivers share the passes of nd_phases.cuh:
//  * k_fused<P, T, MODE>: one CTA owns one replica for a whole launch.  The
//    half spectrum, the stage magnetisation and the FFT scratch live in shared
//    memory; a launch runs n_steps full time steps (RK4: four field
//    evaluations per step, Heun: two) without touching the spectrum in HBM.
//    Used when the CTA's shared-memory footprint fits (P <= 128 in FP32).
//  * k_g_*: the same passes as separate grid-wide kernels with the spectrum
//    in global memory, for the large padded grids (P = 256..1024) and FP64 at
//    P = 128.
// The LLG right-hand side, the RK4 combine, the stochastic Heun predictor and
// corrector with Philox noise and the |m| = 1 renormalisation are fused into
// the epilogue that consumes the inverse transform.
#pragma once
#include "nd_kernels.h"
#include "nd_phases.cuh"
#include "nd_schedule.h"

namespace nd {

// ------------------------------------------------------------- epilogue

template <typename T> __device__ __forceinline__ vec3<T> v3(T x, T y, T z) { return {x, y, z}; }
template <typename T> __device__ __forceinline__ vec3<T> cross3(vec3<T> a, vec3<T> b)
{
    return {fm(a.y, b.z, -(a.z * b.y)), fm(a.z, b.x, -(a.x * b.z)), fm(a.x, b.y, -(a.y * b.x))};
}
template <typename T> __device__ __forceinline__ vec3<T> axpy3(T s, vec3<T> a, vec3<T> b)
{
    return {fm(s, a.x, b.x), fm(s, a.y, b.y), fm(s, a.z, b.z)};
}
template <typename T> __device__ __forceinline__ T dot3(vec3<T> a, vec3<T> b)
{
    return fm(a.z, b.z, fm(a.y, b.y, a.x * b.x));
}
template <typename T> __device__ __forceinline__ vec3<T> normalize3(vec3<T> v)
{
    T r = drsqrt<T>(dot3(v, v));
    return {v.x * r, v.y * r, v.z * r};
}
// Landau-Lifshitz right-hand side m x b - alpha m x (m x b) (Section III.A).
template <typename T> __device__ __forceinline__ vec3<T> llg_rhs(vec3<T> m, vec3<T> b, T alpha)
{
    vec3<T> p = cross3(m, b), q = cross3(m, p);
    return axpy3(-alpha, q, p);
}
// One Heun stage change m x [g - alpha m x g], g = b dtau + sigma w (Section III.C).
template <typename T> __device__ __forceinline__ vec3<T> heun_dm(vec3<T> m, vec3<T> g, T alpha)
{
    vec3<T> p = cross3(m, g);
    return cross3(m, axpy3(-alpha, p, g));
}

// Programmatic dependent launch: the global path's kernels are launched so
// that each may start while its predecessor in the stream drains; before it
// reads anything the predecessor wrote (or the parameter blocks) it waits
// here until that grid has completed and its writes are visible.  Without
// the launch attribute this is a no-op.
__device__ __forceinline__ void wait_prior_grid() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// A stepping call whose final state has a non-finite cell sets the NaN bit of
// the status word.  The cluster kernel looks at the cells it writes last; the
// others are followed by a scan of its own (k_check_finite, 5-10 us): the same
// look took registers from k_fused's column pass (256 replicas, 50 Heun steps:
// 3.44 -> 3.55 ms) and from the global epilogue (8 of D = 500: 5.05 -> 5.10 ms).
template <typename T> __device__ __forceinline__ bool finite3(vec3<T> v)
{
    return isfinite(v.x) && isfinite(v.y) && isfinite(v.z);
}
__device__ __forceinline__ void flag_nan(bool bad, unsigned *status)
{
    if (bad && status) atomicOr(status, ND_DEV_NAN);
}

template <typename T> struct V3Ptr {
    T *p;
    long long s;  // component stride
    __device__ __forceinline__ vec3<T> ld(long long i) const { return {p[i], p[s + i], p[2 * s + i]}; }
    // bypassing L1: for data another CTA may have written during this launch
    __device__ __forceinline__ vec3<T> ldcg(long long i) const
    {
        return {__ldcg(p + i), __ldcg(p + s + i), __ldcg(p + 2 * s + i)};
    }
    __device__ __forceinline__ void st(long long i, vec3<T> v) const { p[i] = v.x; p[s + i] = v.y; p[2 * s + i] = v.z; }
};

// The per-cell update of one stepping stage (Section III.A RK4, Section III.C
// Heun), as a function of the cell's stage input m, its induction b, y_n and
// the stage accumulator a (read by stages > 0) and, for Heun, the normals w:
// returns the next stage's input; acc_new and the flags say what else the
// stage writes (the accumulator, and y_n after the last stage).  Every path
// (on chip, global, fused row pass) calls this one definition, so all of them
// round identically.
template <typename T> struct StageOut {
    vec3<T> nm, acc;
    bool w_acc, w_yn;
};

template <typename T, int MODE>
__device__ __forceinline__ StageOut<T> stage_update(const StepParams<T> &sp, bool noise, int stage, vec3<T> m,
                                                    vec3<T> b, vec3<T> y, vec3<T> a, vec3<T> w)
{
    const T alpha = sp.alpha, dt = sp.dtau;
    StageOut<T> o;
    if (MODE == M_RK4) {
        vec3<T> k = llg_rhs(m, b, alpha);
        if (stage == 0) {
            o.acc = k;
            o.nm = axpy3(T(0.5) * dt, k, m);
            o.w_acc = true; o.w_yn = false;
        } else if (stage < 3) {
            o.acc = axpy3(T(2), k, a);
            o.nm = axpy3(stage == 1 ? T(0.5) * dt : dt, k, y);
            o.w_acc = true; o.w_yn = false;
        } else {
            vec3<T> s = {a.x + k.x, a.y + k.y, a.z + k.z};
            o.nm = normalize3(axpy3(dt / T(6), s, y));
            o.w_acc = false; o.w_yn = true;
        }
    } else {   // M_HEUN
        vec3<T> g = {b.x * dt, b.y * dt, b.z * dt};
        if (noise) g = axpy3(sp.sigma, w, g);
        vec3<T> d = heun_dm(m, g, alpha);
        if (stage == 0) {
            o.acc = d;
            o.nm = normalize3(vec3<T>{m.x + d.x, m.y + d.y, m.z + d.z});
            o.w_acc = true; o.w_yn = false;
        } else {
            o.nm = normalize3(axpy3(T(0.5), vec3<T>{a.x + d.x, a.y + d.y, a.z + d.z}, y));
            o.w_acc = false; o.w_yn = true;
        }
    }
    return o;
}

// Per-cell epilogue of one field evaluation.
//   ms  : stage magnetisation (read; overwritten with the next stage's input)
//   yn  : state y_n (user buffer), acc : stage accumulator (scratch)
//   b   : the full dimensionless induction b_i at this cell
// For Heun, wbuf (when not null) keeps the predictor's normals for the
// corrector, which then reads them instead of regenerating them.
// ynl, accl: where y_n and the accumulator are read from (the same arrays, or
// copies of them staged in shared memory); writes always go to yn and acc.
template <typename T, int MODE>
__device__ __forceinline__ void epilogue_cell(const Replica &r, int cell, long long si, long long mi, vec3<T> b,
                                                V3Ptr<T> ms, V3Ptr<T> yn, V3Ptr<T> acc, V3Ptr<T> out, int stage,
                                                unsigned long long step, V3Ptr<T> wbuf, V3Ptr<T> ynl, V3Ptr<T> accl)
{
    vec3<T> m = ms.ld(mi);
    if (MODE == M_FIELD) {
        out.st(si, b);
    } else if (MODE == M_RK4 || MODE == M_HEUN) {
        const StepParams<T> sp = step_params<T>(r);
        const vec3<T> zero = {T(0), T(0), T(0)};
        vec3<T> y = zero, a = zero, w = zero;
        if (stage > 0) { a = accl.ld(si); y = ynl.ld(si); }
        const bool noise = MODE == M_HEUN && (r.flags & 1);
        if (noise) {
            if (wbuf.p && stage == 1) {
                w = wbuf.ld(mi);
            } else {
                w = thermal_normals<T>(r.seed, (uint32_t)cell, step);
                if (wbuf.p) wbuf.st(mi, w);
            }
        }
        const StageOut<T> o = stage_update<T, MODE>(sp, noise, stage, m, b, y, a, w);
        if (o.w_acc) acc.st(si, o.acc);
        if (o.w_yn) yn.st(si, o.nm);
        ms.st(mi, o.nm);
    }
}

template <typename T, int MODE>
__device__ __forceinline__ void epilogue_cell(const Replica &r, int cell, long long si, long long mi, vec3<T> b,
                                                V3Ptr<T> ms, V3Ptr<T> yn, V3Ptr<T> acc, V3Ptr<T> out, int stage,
                                                unsigned long long step, V3Ptr<T> wbuf = V3Ptr<T>{nullptr, 0})
{
    epilogue_cell<T, MODE>(r, cell, si, mi, b, ms, yn, acc, out, stage, step, wbuf, yn, acc);
}

template <int MODE> struct ModeStages { static constexpr int n = 1; };
template <> struct ModeStages<M_RK4> { static constexpr int n = 4; };
template <> struct ModeStages<M_HEUN> { static constexpr int n = 2; };

// Threads per CTA of the passes whose work divides by warps.  FP64 issues one
// warp instruction per sub-partition in 64-76 cycles, so its CTAs are small: one
// or two warps land on every sub-partition of the chip instead of eight on a few
// SMs (FP64 relaxation of R = 30/65/100 nm, two replicas each: 194 -> 142 ms,
// against rows of 34 us, a reduction of 19 and an update of 11 with 256 threads;
// one FP64 disk of R = 50 nm on this path: 282 -> 137 us per evaluation).
template <typename T> struct GlobNT { static constexpr int v = sizeof(T) == 8 ? 32 : 256; };
template <typename T> struct CellNT { static constexpr int v = sizeof(T) == 8 ? 64 : 256; };
template <typename T> struct RedNT { static constexpr int v = sizeof(T) == 8 ? 128 : 256; };   // partial sums

// ------------------------------------------------------------ fused path

template <int P, typename T>
__host__ __device__ __forceinline__ size_t fused_smem_bytes(int D, int Dpad, int nthreads, bool wbuf = false)
{
    using Gm = FFTGeom<P>;
    size_t tw = sizeof(cplx<T>) * Gm::R1 * Gm::G;
    size_t spec = sizeof(cplx<T>) * 3 * (size_t)D * SpecGeom<P>::RS;
    size_t scr = sizeof(cplx<T>) * (size_t)(nthreads / Gm::G) * Gm::SCRATCH;
    size_t ms = sizeof(T) * 3 * (size_t)D * Dpad;
    size_t w = wbuf ? sizeof(T) * 3 * (size_t)D * Dpad : 0;
    return tw + spec + scr + ms + w;
}

// The hand-over word of a replica: 0, then a count that the signalling segment
// posts every 64 steps, at last kHandedOver.
constexpr int kHandedOver = -1;
__device__ __forceinline__ void post_progress(int *flag, long long n)
{
    if ((n & 63) == 63) atomicExch(flag, (int)((n >> 6) & 0x3fffffff) + 1);
}

// Wait of one thread until another CTA (cluster) of the same launch, one that
// runs already, hands a replica over.  The wait lasts as long as the other
// side works, which grows with the steps of the call and with the difference
// of the replicas' costs: it gives up, and returns false, after `polls` polls
// in which the word has not moved (2^22, about two seconds, against 64 steps of
// at most a few hundred us each).
__device__ __forceinline__ bool wait_flag(int *flag, int polls)
{
    int seen = 0;
    for (int it = 0; it < polls; ++it) {
        const int v = atomicAdd(flag, 0);
        if (v == kHandedOver) {
            __threadfence();
            return true;
        }
        if (v != seen) {
            seen = v;
            it = 0;
        }
        __nanosleep(256);
    }
    return false;
}

template <typename T> __device__ __forceinline__ T warp_sum_t(T v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
template <typename T> __device__ __forceinline__ T warp_max_t(T v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = max(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

// One alignment of the constrained relaxation for a cell (reading of the
// Lagrange-constrained local alignment of Sec. IV): e = b + fictitious field,
// m' = normalise((1-eta) m + eta e/|e|); accumulates the constraint values
// and the exact 2x2 Jacobian of C(m'(lambda)) for cells of the window.
template <typename T> struct RelaxAcc { T C0, C1, J00, J01, J11, res; };

// The field is b + z m; z, a multiple of m that turns nothing, is left out of
// the torque (0 where the caller's b holds all of the field).
template <typename T>
__device__ __forceinline__ vec3<T> relax_cell(vec3<T> m, vec3<T> b, bool inW, T dx, T dy, T l0, T l1, T eta,
                                              RelaxAcc<T> &acc, T z = T(0))
{
    vec3<T> f = b;
    if (inW) f.z = fm(l0 * T(2) * m.z, dx, fm(l1 * T(2) * m.z, dy, f.z));
    const vec3<T> e = axpy3(z, m, f);
    const T en = dsqrt<T>(dot3(e, e));
    const vec3<T> u = {e.x / en, e.y / en, e.z / en};
    const vec3<T> tq = cross3(m, f);
    acc.res = max(acc.res, dsqrt<T>(dot3(tq, tq)) / en);
    const T om = T(1) - eta;
    const vec3<T> v = {fm(eta, u.x, om * m.x), fm(eta, u.y, om * m.y), fm(eta, u.z, om * m.z)};
    const T vn = dsqrt<T>(dot3(v, v));
    const vec3<T> mp = {v.x / vn, v.y / vn, v.z / vn};
    if (inW) {
        const vec3<T> q = {-u.x * u.z / en, -u.y * u.z / en, fm(-u.z, u.z, T(1)) / en};
        const T mq = dot3(mp, q);
        const T kap = eta * fm(-mp.z, mq, q.z) / vn;
        const T w = T(4) * mp.z * m.z * kap;
        acc.C0 = fm(mp.z * mp.z, dx, acc.C0);
        acc.C1 = fm(mp.z * mp.z, dy, acc.C1);
        acc.J00 = fm(w * dx, dx, acc.J00);
        acc.J01 = fm(w * dx, dy, acc.J01);
        acc.J11 = fm(w * dy, dy, acc.J11);
    }
    return mp;
}

// Thread counts of the fused kernel per padded size: variant 0 is the default
// (and the only one of the field, energy and relaxation modes); the stepping
// modes also have the alternatives the autotuner (nd_autotune) times.
template <int P, int V> struct NTV { static constexpr int v = 0; };
template <> struct NTV<128, 0> { static constexpr int v = 512; };
template <> struct NTV<128, 1> { static constexpr int v = 384; };
template <> struct NTV<64, 0> { static constexpr int v = 384; };
template <> struct NTV<64, 1> { static constexpr int v = 256; };
template <> struct NTV<64, 2> { static constexpr int v = 512; };
template <> struct NTV<32, 0> { static constexpr int v = 256; };
template <> struct NTV<32, 1> { static constexpr int v = 128; };
template <> struct NTV<16, 0> { static constexpr int v = 128; };
template <> struct NTV<16, 1> { static constexpr int v = 64; };
template <int P> struct FusedNT { static constexpr int v = NTV<P, 0>::v; };

// Minimum resident CTAs the compiler must allow: the default thread count
// keeps the whole register file for one CTA; the smaller variants are compiled
// lean (up to 512 threads per SM resident) so that several CTAs can share an SM.
template <int P, int NT> struct FusedMinBlocks {
    static constexpr int v = (NT == NTV<P, 0>::v || NT >= 512) ? 1 : 512 / NT;
};

template <int P, typename T, int MODE, int NT>
__global__ void __launch_bounds__(NT, (FusedMinBlocks<P, NT>::v))
    k_fused(const Replica *__restrict__ reps, const int *__restrict__ work, T *__restrict__ ybase,
            T *__restrict__ accbase, T *__restrict__ outbase, const cplx<T> *__restrict__ twP, long long nsteps, unsigned long long step_base,
            RelaxIO *__restrict__ rio, double eta_d, double tol_d, double rc2_d, int max_iter,
            const Segment *__restrict__ segs, const int *__restrict__ seg_off, int *__restrict__ flags,
            int wait_polls, unsigned *__restrict__ status, int use_wbuf)
{
    using Gm = FFTGeom<P>;
    constexpr int G = Gm::G, R1 = Gm::R1, RS = SpecGeom<P>::RS, GPW = Gm::GROUPS_PER_WARP;
    constexpr int NW = NT / 32, NGRP = NT / G;
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ Replica r_sh;   // the descriptor stays in shared memory, not in registers
    __shared__ T lam_s[2];
    __shared__ int conv_s, ok_s, signal_s;
    __shared__ RelaxAcc<T> racc[NW];
    const int tid = threadIdx.x, warp = tid >> 5;
    GroupId<P> gid(tid);
    const int gw = gid.group % GPW;
    constexpr int ncol = P / 2;

    cplx<T> *tw = reinterpret_cast<cplx<T> *>(smem);
    load_twiddles<P>(tw, twP, tid, NT);

    const int s_begin = segs ? seg_off[2 * blockIdx.x] : 0, s_end = segs ? seg_off[2 * blockIdx.x + 1] : 1;
    for (int sg = s_begin; sg < s_end; ++sg) {
        int ridx, wait = 0, signal = 0;
        long long sbeg = 0, nseg = nsteps;
        if (segs) {
            const Segment g = segs[sg];
            ridx = g.rep; wait = g.wait; signal = g.signal; sbeg = g.step_begin; nseg = g.nsteps;
        } else {
            ridx = work[blockIdx.x];
        }
        if (tid == 0) {
            ok_s = wait ? (int)wait_flag(flags + ridx, wait_polls) : 1;
            if (!ok_s) atomicOr(status, ND_DEV_TIMEOUT);
            signal_s = signal;
            r_sh = reps[ridx];
        }
        __syncthreads();
        if (!ok_s) break;
        const Replica &r = r_sh;
        const int D = r.D, Dpad = r.Dpad, DD = D * D;
        const long long cs = (long long)D * RS;           // spectrum component stride
        const long long ms_s = (long long)D * Dpad;       // stage-state component stride
        cplx<T> *spec = tw + R1 * G;
        cplx<T> *scratch = spec + 3 * cs;
        T *msm = reinterpret_cast<T *>(scratch + NGRP * Gm::SCRATCH);
        T *wsm = use_wbuf ? msm + 3 * ms_s : nullptr;
        cplx<T> *scr = scratch + gid.group * Gm::SCRATCH;

        V3Ptr<T> yn{ybase + r.state_off, ms_s};
        V3Ptr<T> acc{accbase ? accbase + r.state_off : nullptr, ms_s};
        V3Ptr<T> out{outbase ? outbase + r.state_off : nullptr, ms_s};
        V3Ptr<T> ms{msm, ms_s};
        V3Ptr<T> wb{wsm, ms_s};
        for (int cell = tid; cell < DD; cell += NT) {
            const int y = cell / D, x = cell - y * D;
            const long long si = (long long)y * Dpad + x;
            vec3<T> v = r.mask[cell] ? yn.ldcg(si) : vec3<T>{T(0), T(0), T(0)};   // may come from another CTA
            ms.st(si, v);
        }
        __syncthreads();

        // row tasks: one real row each (half-length transforms) at P = 128,
        // else a complex row pair each
        constexpr bool HR = HalfRows<P>::on;
        const int nrow = row_pass_tasks<P>(D);
        T relX = 0, relY = 0;
        if (MODE == M_RELAX) {
            relX = (T)rio[ridx].X[0];
            relY = (T)rio[ridx].X[1];
            if (tid == 0) { lam_s[0] = (T)rio[ridx].lam[0]; lam_s[1] = (T)rio[ridx].lam[1]; conv_s = 0; }
            __syncthreads();
        }
        const long long nst = MODE == M_FIELD ? 1 : (MODE == M_RELAX ? (long long)max_iter : nseg);
        long long n = 0;
        T res_last = T(0);
        for (n = 0; n < nst; ++n) {
            for (int stage = 0; stage < ModeStages<MODE>::n; ++stage) {
                for (int qb = warp * GPW; qb < nrow; qb += NW * GPW) {
                    const int q = qb + gw;
                    if constexpr (HR) {
                        const int c = q / D, y = q - c * D;
                        const bool act = q < nrow;
                        const int cc = act ? c : 0, yy = act ? y : 0;
                        row_fwd_half<P, T>(act, msm + cc * ms_s + (long long)yy * Dpad, D,
                                           spec + cc * cs + (long long)yy * RS, gid.t, scr, tw, gid.gmask);
                    } else {
                        row_fwd_task<P, T>(q, q < nrow, D, msm, Dpad, ms_s, spec, cs, gid.t, gid.lane, scr, tw,
                                           gid.gmask);
                    }
                }
                __syncthreads();
                for (int qb = warp * GPW; qb < ncol; qb += NW * GPW) {
                    const int q = qb + gw;
                    col_task<P, T>(q, q < ncol, D, spec, cs, reinterpret_cast<const T *>(r.Ghat), gid.t, gid.lane,
                                   scr, tw, gid.gmask);
                }
                __syncthreads();
                for (int qb = warp * GPW; qb < nrow; qb += NW * GPW) {
                    const int q = qb + gw;
                    if constexpr (HR) {
                        const int c = q / D, y = q - c * D;
                        const bool act = q < nrow;
                        const int cc = act ? c : 0, yy = act ? y : 0;
                        cplx<T> *row = spec + cc * cs + (long long)yy * RS;
                        row_inv_half<P, T>(act, row, D, reinterpret_cast<T *>(row), gid.t, scr, tw, gid.gmask);
                    } else {
                        row_inv_task<P, T>(q, q < nrow, D, spec, cs, gid.t, scr, tw, gid.gmask);
                    }
                }
                __syncthreads();
                const T *hr = reinterpret_cast<const T *>(spec);
                const StepParams<T> sp = step_params<T>(r);
                if (MODE == M_RELAX) {
                    // sweep: trial alignment with the current multipliers, reductions
                    const T eta = (T)eta_d, rc2 = (T)rc2_d, l0 = lam_s[0], l1 = lam_s[1];
                    RelaxAcc<T> a = {T(0), T(0), T(0), T(0), T(0), T(0)};
                    for (int cell = tid; cell < DD; cell += NT) {
                        if (!r.mask[cell]) continue;
                        const int y = cell / D, x = cell - y * D;
                        const long long si = (long long)y * Dpad + x, hi = (long long)y * (2 * RS) + x;
                        vec3<T> b = {hr[hi] + sp.chext[0], hr[2 * cs + hi] + sp.chext[1], hr[4 * cs + hi] + sp.chext[2]};
                        const T dx = (T)x - T(0.5) * (T)(D - 1) - relX, dy = (T)y - T(0.5) * (T)(D - 1) - relY;
                        relax_cell<T>(ms.ld(si), b, fm(dx, dx, dy * dy) < rc2, dx, dy, l0, l1, eta, a);
                    }
                    a.C0 = warp_sum_t(a.C0); a.C1 = warp_sum_t(a.C1); a.J00 = warp_sum_t(a.J00);
                    a.J01 = warp_sum_t(a.J01); a.J11 = warp_sum_t(a.J11); a.res = warp_max_t(a.res);
                    if ((tid & 31) == 0) racc[warp] = a;
                    __syncthreads();
                    if (tid == 0) {
                        RelaxAcc<T> s = racc[0];
                        for (int w = 1; w < NW; ++w) {
                            s.C0 += racc[w].C0; s.C1 += racc[w].C1; s.J00 += racc[w].J00; s.J01 += racc[w].J01;
                            s.J11 += racc[w].J11; s.res = max(s.res, racc[w].res);
                        }
                        res_last = s.res;
                        if (s.res < (T)tol_d) {
                            conv_s = 1;
                        } else {
                            const T det = s.J00 * s.J11 - s.J01 * s.J01;
                            if (det != T(0) && isfinite(det)) {
                                lam_s[0] += -(s.J11 * s.C0 - s.J01 * s.C1) / det;
                                lam_s[1] += -(-s.J01 * s.C0 + s.J00 * s.C1) / det;
                            }
                        }
                    }
                    __syncthreads();
                    if (conv_s) break;   // leaves the stage loop; the step loop stops below
                    const T m0 = lam_s[0], m1 = lam_s[1];
                    for (int cell = tid; cell < DD; cell += NT) {
                        if (!r.mask[cell]) continue;
                        const int y = cell / D, x = cell - y * D;
                        const long long si = (long long)y * Dpad + x, hi = (long long)y * (2 * RS) + x;
                        vec3<T> b = {hr[hi] + sp.chext[0], hr[2 * cs + hi] + sp.chext[1], hr[4 * cs + hi] + sp.chext[2]};
                        const T dx = (T)x - T(0.5) * (T)(D - 1) - relX, dy = (T)y - T(0.5) * (T)(D - 1) - relY;
                        RelaxAcc<T> dummy = {T(0), T(0), T(0), T(0), T(0), T(0)};
                        ms.st(si, relax_cell<T>(ms.ld(si), b, fm(dx, dx, dy * dy) < rc2, dx, dy, m0, m1, eta, dummy));
                    }
                    __syncthreads();
                    continue;
                }
                const unsigned long long step = step_base + r.step0 + (unsigned long long)(sbeg + n);
                // Stages that read y_n and the accumulator get both copied, with
                // 16-byte loads all in flight at once, into the FFT scratch (idle
                // during the epilogue) instead of two dependent round trips to L2
                // per cell.
                V3Ptr<T> ynl = yn, accl = acc;
                if ((MODE == M_HEUN && stage == 1) || (MODE == M_RK4 && stage > 0)) {
                    const long long words = 3 * ms_s * (long long)sizeof(T) / 16;   // Dpad is a multiple of 4
                    const bool fits = 2 * words * 16 <= (long long)(NGRP * Gm::SCRATCH * sizeof(cplx<T>));
                    const bool aligned = ((reinterpret_cast<uintptr_t>(yn.p) | reinterpret_cast<uintptr_t>(acc.p)) & 15) == 0;
                    if (fits && aligned) {
                        int4 *dst = reinterpret_cast<int4 *>(scratch);
                        const int4 *gy = reinterpret_cast<const int4 *>(yn.p), *ga = reinterpret_cast<const int4 *>(acc.p);
                        for (long long i = tid; i < words; i += NT) {
                            const int4 u = __ldcg(gy + i), v = __ldcg(ga + i);
                            dst[i] = u;
                            dst[words + i] = v;
                        }
                        __syncthreads();
                        ynl = V3Ptr<T>{reinterpret_cast<T *>(scratch), ms_s};
                        accl = V3Ptr<T>{reinterpret_cast<T *>(scratch) + 3 * ms_s, ms_s};
                    }
                }
                // the external field of this step (a scheduled one in the stepping modes)
                const vec3<T> cx = (MODE == M_RK4 || MODE == M_HEUN) ? step_chext<T>(r, sp, step)
                                                                     : vec3<T>{sp.chext[0], sp.chext[1], sp.chext[2]};
                if (MODE == M_FIELD) {   // the whole output block, zero outside the disk
                    for (int i = tid; i < D * Dpad; i += NT) {
                        const int y = i / Dpad, x = i - y * Dpad;
                        const long long hi = (long long)y * (2 * RS) + x;
                        const bool in = x < D && r.mask[y * D + x];
                        out.st(i, in ? vec3<T>{hr[hi] + cx.x, hr[2 * cs + hi] + cx.y, hr[4 * cs + hi] + cx.z}
                                     : vec3<T>{T(0), T(0), T(0)});
                    }
                    continue;
                }
                // over the disk's cells only (a compacted list), so that no warp
                // spends an iteration on cells outside the disk
                for (int k = tid; k < r.ncells; k += NT) {
                    const int cell = __ldg(r.cells + k);
                    const int y = cell / D, x = cell - y * D;
                    const long long si = (long long)y * Dpad + x;
                    const long long hi = (long long)y * (2 * RS) + x;
                    vec3<T> b = {hr[hi] + cx.x, hr[2 * cs + hi] + cx.y, hr[4 * cs + hi] + cx.z};
                    epilogue_cell<T, MODE>(r, cell, si, si, b, ms, yn, acc, out, stage, step, wb, ynl, accl);
                }
                __syncthreads();
            }
            if ((MODE == M_RK4 || MODE == M_HEUN) && tid == 0 && signal_s) post_progress(flags + ridx, n);
            if (MODE == M_RELAX && conv_s) break;
        }
        if (MODE == M_RELAX) {
            // the relaxed state back to the caller's buffer
            for (int cell = tid; cell < DD; cell += NT) {
                if (!r.mask[cell]) continue;
                const int y = cell / D, x = cell - y * D;
                const long long si = (long long)y * Dpad + x;
                yn.st(si, ms.ld(si));
            }
            if (tid == 0) {
                rio[ridx].lam[0] = (double)lam_s[0];
                rio[ridx].lam[1] = (double)lam_s[1];
                rio[ridx].resid = (double)res_last;
                rio[ridx].iters = (int)n;
                rio[ridx].status = conv_s ? 0 : 1;
            }
        }
        __syncthreads();   // every write of this segment is done before the flag and the next segment
        if (tid == 0 && signal_s) {
            __threadfence();
            atomicExch(flags + ridx, kHandedOver);
        }
    }
}

// ----------------------------------------------------------- global path

// Resident CTAs per SM the row passes are compiled for: at P = 1024 (FP32) a
// cap of 80 registers leaves room for three CTAs of 256 threads, which the
// latency-bound row loads need.
template <int P, typename T> struct RowsMinB { static constexpr int v = (P == 1024 && sizeof(T) == 4) ? 3 : 1; };
template <int P, typename T, int NT>
__global__ void __launch_bounds__(NT, RowsMinB<P, T>::v)
    k_g_rows(const Replica *__restrict__ reps, const int *__restrict__ work, const T *__restrict__ msbase,
             cplx<T> *__restrict__ specbase, const cplx<T> *__restrict__ twP, int inverse)
{
    using Gm = FFTGeom<P>;
    constexpr int G = Gm::G, R1 = Gm::R1, RS = SpecGeom<P>::RS, NGRP = groups_per_block<P, NT>();
    extern __shared__ __align__(16) unsigned char gsm[];
    cplx<T> *tw = reinterpret_cast<cplx<T> *>(gsm);
    cplx<T> *scratch = tw + R1 * G;
    const int tid = threadIdx.x;
    load_twiddles<P>(tw, twP, tid, NT);   // constant: before the wait
    wait_prior_grid();
    const Replica r = reps[work[blockIdx.y]];
    const int D = r.D;
    __syncthreads();
    GroupId<P> gid(tid);
    const int q = blockIdx.x * NGRP + gid.group;
    const int nrow = row_pass_tasks<P>(D);
    if (blockIdx.x * NGRP >= nrow) return;   // CTA-uniform
    if (!gid.valid) return;                  // lanes past the warp's last group
    const long long cs = (long long)D * RS;
    cplx<T> *spec = specbase + r.spec_off;
    cplx<T> *scr = scratch + gid.group * Gm::SCRATCH;
    const long long ms_s = (long long)D * r.Dpad;
    if constexpr (HalfRows<P>::on) {
        const bool act = q < nrow;
        const int c = act ? q / D : 0, y = act ? q - c * D : 0;
        cplx<T> *row = spec + c * cs + (long long)y * RS;
        if (!inverse)
            row_fwd_half<P, T>(act, msbase + r.state_off + c * ms_s + (long long)y * r.Dpad, D, row, gid.t, scr, tw,
                               gid.gmask);
        else
            row_inv_half<P, T>(act, row, D, reinterpret_cast<T *>(row), gid.t, scr, tw, gid.gmask);
    } else if (!inverse) {
        row_fwd_task<P, T>(q, q < nrow, D, msbase + r.state_off, r.Dpad, ms_s, spec, cs, gid.t, gid.lane, scr, tw,
                           gid.gmask);
    } else {
        row_inv_task<P, T, true>(q, q < nrow, D, spec, cs, gid.t, scr, tw, gid.gmask);
    }
}

template <int P, typename T, int NT>
__global__ void __launch_bounds__(NT)
    k_g_cols(const Replica *__restrict__ reps, const int *__restrict__ work, cplx<T> *__restrict__ specbase,
             const cplx<T> *__restrict__ twP)
{
    using Gm = FFTGeom<P>;
    constexpr int G = Gm::G, R1 = Gm::R1, RS = SpecGeom<P>::RS, NGRP = groups_per_block<P, NT>();
    extern __shared__ __align__(16) unsigned char gsm[];
    cplx<T> *tw = reinterpret_cast<cplx<T> *>(gsm);
    cplx<T> *scratch = tw + R1 * G;
    const int tid = threadIdx.x;
    load_twiddles<P>(tw, twP, tid, NT);   // constant: before the wait
    wait_prior_grid();
    const Replica r = reps[work[blockIdx.y]];
    const int D = r.D;
    __syncthreads();
    GroupId<P> gid(tid);
    if (!gid.valid) return;   // lanes past the warp's last group
    const int q = blockIdx.x * NGRP + gid.group;
    const long long cs = (long long)D * RS;
    col_task<P, T>(q, q < P / 2, D, specbase + r.spec_off, cs, reinterpret_cast<const T *>(r.Ghat), gid.t, gid.lane,
                   scratch + gid.group * Gm::SCRATCH, tw, gid.gmask);
}

// Tiled column pass for the large grids.  A CTA of eight FFT groups takes one
// of two kinds of task: four adjacent columns of the x and y components (group
// 4c + j holds component c of column kx0 + j, its partner for the in-plane
// tensor is group ^ 4), or eight adjacent columns of z.  Both cost about the
// same, and one launch runs the xy tasks of all replicas and then the z tasks:
// as two launches (xy; z with four groups) each pass ended in a round that
// filled part of the SMs (24 replicas of D = 121 at P = 256: 18.0 + 10.6 us, 768
// tasks each on 608 resident CTAs; 8 of D = 500 at P = 1024: 55.8 + 27.3 us).
// The task's tiles [D][4] x 2 or [D][8] move between the spectrum and the
// groups' scratch areas as row-contiguous runs of four or eight complex words
// (whole 32-byte sectors: rows start on sectors, SpecGeom::RS).  The packed
// real columns kx = 0, P/2 are column 0 of the first block.  Persistent grid.
template <int P, typename T> struct ColTile {
    static constexpr int G = FFTGeom<P>::G;
    static constexpr int NG = 8;
    // whole warps: with ten-lane groups (P = 200, three to a warp) three warps
    // with one group slot and each warp's last two lanes idle
    static constexpr bool POW2 = FFTGeom<P>::POW2;
    static constexpr int GPW = FFTGeom<P>::GROUPS_PER_WARP;
    static constexpr int NT = POW2 ? NG * G : (NG + GPW - 1) / GPW * 32;
    static constexpr int NXY = P / 2 / 4;                // xy tasks of a replica
    static constexpr int NZ = (P / 2 + 7) / 8;           // its z tasks
    // resident CTAs per SM the kernel is compiled for: 16 warps at 128
    // registers (FP64 columns take twice the registers)
    static constexpr int MINB = sizeof(T) == 8 ? 1 : 512 / NT;
    // How the packed pair is transformed.  With 32 points per thread (P = 512,
    // 1024) a second inlined transform for it pushes the kernel past its 128
    // registers (96-124 bytes of spills per thread in FP32), so the pair moves
    // through the tile like the other columns and runs the same transform
    // calls; with 16 or 24 points per thread nothing spills, and the pair
    // loads, transforms and stores its two columns itself, which measured 3%
    // faster at P = 256.
    static constexpr bool SHARED_PACKED = FFTGeom<P>::R1 >= 32;
};

template <int P, typename T>
__global__ void __launch_bounds__(ColTile<P, T>::NT, ColTile<P, T>::MINB)
    k_g_cols_tile(const Replica *__restrict__ reps, const int *__restrict__ work, int nwork,
                  cplx<T> *__restrict__ specbase, const cplx<T> *__restrict__ twP)
{
    using Gm = FFTGeom<P>;
    using CT = ColTile<P, T>;
    constexpr int G = Gm::G, R1 = Gm::R1, KH = SpecGeom<P>::KH, RS = SpecGeom<P>::RS, NT = CT::NT, SCR = Gm::SCRATCH;
    constexpr bool SP = CT::SHARED_PACKED;
    static_assert(RS % 4 == 0, "rows start on 32-byte sectors");
    extern __shared__ __align__(16) unsigned char gsm[];
    cplx<T> *tw = reinterpret_cast<cplx<T> *>(gsm);
    cplx<T> *scratch = tw + R1 * G;
    const int tid = threadIdx.x;
    load_twiddles<P>(tw, twP, tid, NT);   // constant: before the wait
    wait_prior_grid();
    GroupId<P> gid(tid);
    const int g = gid.group, t = gid.t;
    // a group of the block (idle slots and lanes take part in the tile moves
    // and the barriers only)
    const bool gv = CT::POW2 || (gid.valid && g < CT::NG);
    cplx<T> *scr = scratch + g * SCR;
    const cplx<T> *other = scratch + (g ^ 4) * SCR;   // xy tasks only
    const int jj = tid & 7;                            // the tile moves: this thread's column of the task
    const int nxy = nwork * CT::NXY, ntask = nxy + nwork * CT::NZ;
    for (int task = blockIdx.x; task < ntask; task += gridDim.x) {
        const bool xy = task < nxy;
        const int ti = xy ? task : task - nxy, per = xy ? CT::NXY : CT::NZ;
        const int wi = ti / per, cb = ti - wi * per, kx0 = (xy ? 4 : 8) * cb;
        const int j = xy ? g & 3 : g, c = xy ? g >> 2 : 2;
        const Replica &r = reps[work[wi]];
        const int D = r.D;
        const long long cs = (long long)D * RS;
        cplx<T> *spec = specbase + r.spec_off;
        const T *Ghat = reinterpret_cast<const T *>(r.Ghat);
        const bool packed = (cb == 0 && j == 0);
        const bool gon = gv && (P % 16 == 0 || kx0 + j < P / 2);   // (the last z task of P = 200 has four columns)
        const int kx = packed || !gon ? 1 : kx0 + j;   // (the packed group reads no kx column of the table)
        // this thread's column in the tile moves: (column 0 of block 0: the
        // packed pair c_0 + i c_{P/2}, when it moves through the tile)
        const int mj = xy ? jj & 3 : jj, mc = xy ? jj >> 2 : 2;
        const bool ppair = cb == 0 && mj == 0, mon = P % 16 == 0 || kx0 + mj < P / 2;
        cplx<T> *const tile = scratch + jj * SCR;
        cplx<T> *const gcol = spec + mc * cs + kx0 + mj;
        __syncthreads();   // twiddles filled / the previous task's tiles stored
        if (mon && (SP || !ppair)) {
            if (SP && ppair) {
                for (int y = tid >> 3; y < D; y += NT / 8)
                    tile[y] = {gcol[(long long)y * RS].x, gcol[(long long)y * RS + P / 2].x};
            } else {
                for (int y = tid >> 3; y < D; y += NT / 8) tile[y] = gcol[(long long)y * RS];
            }
        }
        __syncthreads();
        cplx<T> v[R1];
        if (!gon) {
        } else if (!SP && packed) {
            packed_col_fwd<P, T>(v, c, true, D, spec + c * cs, Ghat, t, gid.lane, scr, tw, gid.gmask);
        } else {
#pragma unroll
            for (int o = 0; o < R1; ++o) v[o] = {T(0), T(0)};
#pragma unroll
            for (int o = 0; o < R1 / 2; ++o) {   // rows >= D (and so >= P/2) are zero padding
                const int y = t + G * o;
                if (y < D) v[o] = scr[y];
            }
            __syncwarp(gid.gmask);
            fft_group<P, -1, FFT_HALF_IN>(v, t, scr, tw, gid.gmask);
            if (xy) {
#pragma unroll
                for (int o = 0; o < R1; ++o) scr[o * G + t] = v[o];
            }
        }
        if (xy) __syncthreads();
        if (!gon) {
        } else if (packed) {
            // (the packed pair's partner is packed too and reads no spectrum of it)
            if (SP) packed_col_scale<P, T>(v, c, Ghat, t, scr, gid.gmask);
        } else {
            // the component-major copy of the table: each group reads only the
            // entries it uses (4 or 8 bytes per point instead of 16)
            constexpr int KK = KH * KH;
            const T *Gs = Ghat + 4 * KK + kx * KH;
            if (xy) {
                const T *gd = Gs + c * KK, *go = Gs + 2 * KK;   // diagonal entry (xx or yy), xy
#pragma unroll
                for (int o = 0; o < R1; ++o) {
                    const int ky = t + G * o;
                    const bool up = ky <= P / 2;
                    const int kyr = up ? ky : P - ky;
                    const T gdiag = __ldg(gd + kyr), gxy0 = __ldg(go + kyr);
                    const T gxy = up ? gxy0 : -gxy0;   // G_xy is odd in ky
                    const cplx<T> w = other[o * G + t];
                    v[o] = c == 0 ? tensor_row(gdiag, v[o], gxy, w) : tensor_row(gxy, w, gdiag, v[o]);
                }
            } else {
                const T *gz = Gs + 3 * KK;
#pragma unroll
                for (int o = 0; o < R1; ++o) {
                    const int ky = t + G * o;
                    const int kyr = ky <= P / 2 ? ky : P - ky;
                    v[o] = cscale(v[o], __ldg(gz + kyr));
                }
            }
        }
        if (xy) __syncthreads();   // the partner's spectrum is read before the scratch is reused
        if (gon) {
            fft_group<P, +1, FFT_HALF_OUT>(v, t, scr, tw, gid.gmask);
            __syncwarp(gid.gmask);
            if (!SP && packed) {
                packed_col_store<P, T>(v, true, D, spec + c * cs, t);
            } else {
#pragma unroll
                for (int o = 0; o < R1 / 2; ++o) {
                    const int y = t + G * o;
                    if (y < D) scr[y] = v[o];
                }
            }
        }
        __syncthreads();
        if (mon && (SP || !ppair)) {
            if (SP && ppair) {
                for (int y = tid >> 3; y < D; y += NT / 8) {
                    const cplx<T> u = tile[y];
                    gcol[(long long)y * RS] = {u.x, T(0)};
                    gcol[(long long)y * RS + P / 2] = {u.y, T(0)};
                }
            } else {
                for (int y = tid >> 3; y < D; y += NT / 8) gcol[(long long)y * RS] = tile[y];
            }
        }
    }
}

// Elementwise epilogue of the global path.  grid = (cell blocks, replicas).
template <int P, typename T, int MODE>
__global__ void __launch_bounds__(CellNT<T>::v)
    k_g_epi(const Replica *__restrict__ reps, const int *__restrict__ work, T *__restrict__ msbase,
            T *__restrict__ ybase, T *__restrict__ accbase, T *__restrict__ outbase,
            const cplx<T> *__restrict__ specbase, int stage, unsigned long long step)
{
    constexpr int RS = SpecGeom<P>::RS;
    const int ridx = work[blockIdx.y];
    const Replica r = reps[ridx];
    const int D = r.D, DD = D * D;
    const long long ms_s = (long long)D * r.Dpad, cs = (long long)D * RS;
    const int cell = blockIdx.x * CellNT<T>::v + threadIdx.x;
    if (cell < DD && r.mask[cell]) {
        const int y = cell / D, x = cell - y * D;
        const long long si = (long long)y * r.Dpad + x;
        const T *hr = reinterpret_cast<const T *>(specbase + r.spec_off);
        const long long hi = (long long)y * (2 * RS) + x;
        const StepParams<T> sp = step_params<T>(r);
        const vec3<T> cx = (MODE == M_RK4 || MODE == M_HEUN) ? step_chext<T>(r, sp, step + r.step0)
                                                             : vec3<T>{sp.chext[0], sp.chext[1], sp.chext[2]};
        vec3<T> b = {hr[hi] + cx.x, hr[2 * cs + hi] + cx.y, hr[4 * cs + hi] + cx.z};
        V3Ptr<T> ms{msbase + r.state_off, ms_s}, yn{ybase + r.state_off, ms_s};
        V3Ptr<T> acc{accbase ? accbase + r.state_off : nullptr, ms_s}, out{outbase ? outbase + r.state_off : nullptr, ms_s};
        epilogue_cell<T, MODE>(r, cell, si, si, b, ms, yn, acc, out, stage, step + r.step0);
    }
}

// Four consecutive elements of a row (16-byte aligned): one 16-byte access in
// FP32, two in FP64.
template <typename T> struct Quad { T v[4]; };
template <typename T> __device__ __forceinline__ Quad<T> ld_quad(const T *p);
template <> __device__ __forceinline__ Quad<float> ld_quad<float>(const float *p)
{
    const float4 a = __ldcg(reinterpret_cast<const float4 *>(p));
    return {{a.x, a.y, a.z, a.w}};
}
template <> __device__ __forceinline__ Quad<double> ld_quad<double>(const double *p)
{
    const double2 a = __ldcg(reinterpret_cast<const double2 *>(p)), b = __ldcg(reinterpret_cast<const double2 *>(p) + 1);
    return {{a.x, a.y, b.x, b.y}};
}
template <typename T> __device__ __forceinline__ void st_quad(T *p, const Quad<T> &q);
template <> __device__ __forceinline__ void st_quad<float>(float *p, const Quad<float> &q)
{
    *reinterpret_cast<float4 *>(p) = make_float4(q.v[0], q.v[1], q.v[2], q.v[3]);
}
template <> __device__ __forceinline__ void st_quad<double>(double *p, const Quad<double> &q)
{
    reinterpret_cast<double2 *>(p)[0] = make_double2(q.v[0], q.v[1]);
    reinterpret_cast<double2 *>(p)[1] = make_double2(q.v[2], q.v[3]);
}

// Epilogue of the global path for the stepping modes with quad access: each
// thread takes four consecutive cells of a row, loads the field rows (the
// spectrum buffer viewed as real rows) and the state rows it needs with
// 16-byte accesses, applies stage_update to the cells inside the disk and
// stores whole quads back (cells outside the disk and padding columns are
// written back unchanged).  grid = (quad blocks, replicas).  Requires 16-byte
// aligned state buffers (rows and replica blocks are multiples of 4
// elements; the spectrum rows start on 32-byte sectors).
template <int P, typename T, int MODE>
__global__ void __launch_bounds__(CellNT<T>::v)
    k_g_epi_quad(const Replica *__restrict__ reps, const int *__restrict__ work, T *__restrict__ msbase,
                 T *__restrict__ ybase, T *__restrict__ accbase, const cplx<T> *__restrict__ specbase, int stage,
                 unsigned long long step)
{
    constexpr int RS = SpecGeom<P>::RS;
    static_assert(RS % 2 == 0, "field rows start on 16-byte boundaries");
    wait_prior_grid();
    const Replica &r = reps[work[blockIdx.y]];
    const int D = r.D, Dpad = r.Dpad, qpr = Dpad / 4;
    const int qd = blockIdx.x * CellNT<T>::v + threadIdx.x;
    if (qd >= D * qpr) return;
    const int y = qd / qpr, x0 = 4 * (qd - y * qpr);
    const long long ms_s = (long long)D * Dpad, cs2 = 2LL * D * RS;   // component strides (state, field rows)
    const long long si = (long long)y * Dpad + x0;
    const T *hr = reinterpret_cast<const T *>(specbase + r.spec_off) + (long long)y * (2 * RS) + x0;
    T *msr = msbase + r.state_off + si, *ynr = ybase + r.state_off + si, *acr = accbase + r.state_off + si;
    unsigned in = 0u;
#pragma unroll
    for (int u = 0; u < 4; ++u)
        if (x0 + u < D && r.mask[y * D + x0 + u]) in |= 1u << u;
    if (!in) return;
    Quad<T> m[3], b[3], yv[3], av[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        m[c] = ld_quad<T>(msr + c * ms_s);
        b[c] = ld_quad<T>(hr + c * cs2);
        if (stage > 0) {
            yv[c] = ld_quad<T>(ynr + c * ms_s);
            av[c] = ld_quad<T>(acr + c * ms_s);
        } else {
            yv[c] = av[c] = Quad<T>{{T(0), T(0), T(0), T(0)}};
        }
    }
    const StepParams<T> sp = step_params<T>(r);
    const bool noise = MODE == M_HEUN && (r.flags & 1);
    const unsigned long long nstep = step + r.step0;
    const vec3<T> cx = step_chext<T>(r, sp, nstep);
    Quad<T> nm[3] = {m[0], m[1], m[2]}, na[3] = {av[0], av[1], av[2]}, ny[3] = {yv[0], yv[1], yv[2]};
    bool w_acc = false, w_yn = false;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        if (!((in >> u) & 1u)) continue;
        const vec3<T> mu = {m[0].v[u], m[1].v[u], m[2].v[u]};
        const vec3<T> bu = {b[0].v[u] + cx.x, b[1].v[u] + cx.y, b[2].v[u] + cx.z};
        const vec3<T> yu = {yv[0].v[u], yv[1].v[u], yv[2].v[u]}, au = {av[0].v[u], av[1].v[u], av[2].v[u]};
        const vec3<T> w = noise ? thermal_normals<T>(r.seed, (uint32_t)(y * D + x0 + u), nstep)
                                : vec3<T>{T(0), T(0), T(0)};
        const StageOut<T> o = stage_update<T, MODE>(sp, noise, stage, mu, bu, yu, au, w);
        nm[0].v[u] = o.nm.x; nm[1].v[u] = o.nm.y; nm[2].v[u] = o.nm.z;
        if (o.w_acc) { na[0].v[u] = o.acc.x; na[1].v[u] = o.acc.y; na[2].v[u] = o.acc.z; w_acc = true; }
        if (o.w_yn) { ny[0].v[u] = o.nm.x; ny[1].v[u] = o.nm.y; ny[2].v[u] = o.nm.z; w_yn = true; }
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        st_quad<T>(msr + c * ms_s, nm[c]);
        if (w_acc) {
            if (stage == 0) {   // the accumulator was not loaded: outside cells keep their (unused) values
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    if ((in >> u) & 1u) acr[c * ms_s + u] = na[c].v[u];
            } else {
                st_quad<T>(acr + c * ms_s, na[c]);
            }
        }
        if (w_yn) st_quad<T>(ynr + c * ms_s, ny[c]);
    }
}

// Copy y_n into the stage buffer (masked), for the global path.
template <typename T>
__global__ void k_g_load_stage(const Replica *__restrict__ reps, const int *__restrict__ work, const T *__restrict__ ybase,
                               T *__restrict__ msbase)
{
    wait_prior_grid();
    const Replica r = reps[work[blockIdx.y]];
    const int D = r.D, DD = D * D;
    const long long ms_s = (long long)D * r.Dpad;
    for (int cell = blockIdx.x * blockDim.x + threadIdx.x; cell < DD; cell += gridDim.x * blockDim.x) {
        const int y = cell / D, x = cell - y * D;
        const long long si = r.state_off + (long long)y * r.Dpad + x;
        const bool in = r.mask[cell];
        for (int c = 0; c < 3; ++c) msbase[si + c * ms_s] = in ? ybase[si + c * ms_s] : T(0);
    }
}

// Constrained relaxation on the global path (Sec. IV; same sweep as the fused
// kernel's relaxation mode): per iteration the field passes, then
//   k_g_relax_reduce  per-block partial sums of the constraint values C_k, the
//                     Jacobian J and the residual max |m x e|/|e| of the trial
//                     alignment with the current multipliers,
//   k_g_relax_newton  per replica: fixed-order total, convergence test, one
//                     Newton step on the multipliers,
//   k_g_relax_update  the damped alignment with the new multipliers.
// Replicas that have converged (status 0) are left untouched.
template <int P, typename T>
__global__ void __launch_bounds__(RedNT<T>::v)
    k_g_relax_reduce(const Replica *__restrict__ reps, const int *__restrict__ work, const T *__restrict__ msbase,
                     const cplx<T> *__restrict__ specbase, const RelaxIO *__restrict__ rio, double rc2_d,
                     double eta_d, double *__restrict__ part)
{
    constexpr int RS = SpecGeom<P>::RS;
    __shared__ RelaxAcc<T> racc[RedNT<T>::v / 32];
    const int ridx = work[blockIdx.y], tid = threadIdx.x;
    if (rio[ridx].status == 0) return;   // CTA-uniform
    const Replica &r = reps[ridx];
    const int D = r.D, DD = D * D;
    const long long ms_s = (long long)D * r.Dpad, cs = (long long)D * RS;
    const T *hr = reinterpret_cast<const T *>(specbase + r.spec_off);
    const V3Ptr<T> ms{const_cast<T *>(msbase) + r.state_off, ms_s};
    const T relX = (T)rio[ridx].X[0], relY = (T)rio[ridx].X[1], l0 = (T)rio[ridx].lam[0], l1 = (T)rio[ridx].lam[1];
    const T eta = (T)eta_d, rc2 = (T)rc2_d;
    const StepParams<T> sp = step_params<T>(r);
    RelaxAcc<T> a = {T(0), T(0), T(0), T(0), T(0), T(0)};
    for (int cell = blockIdx.x * RedNT<T>::v + tid; cell < DD; cell += kRelaxBlocks * RedNT<T>::v) {
        if (!r.mask[cell]) continue;
        const int y = cell / D, x = cell - y * D;
        const long long si = (long long)y * r.Dpad + x, hi = (long long)y * (2 * RS) + x;
        const vec3<T> b = {hr[hi] + sp.chext[0], hr[2 * cs + hi] + sp.chext[1], hr[4 * cs + hi] + sp.chext[2]};
        const T dx = (T)x - T(0.5) * (T)(D - 1) - relX, dy = (T)y - T(0.5) * (T)(D - 1) - relY;
        relax_cell<T>(ms.ld(si), b, fm(dx, dx, dy * dy) < rc2, dx, dy, l0, l1, eta, a);
    }
    a.C0 = warp_sum_t(a.C0); a.C1 = warp_sum_t(a.C1); a.J00 = warp_sum_t(a.J00);
    a.J01 = warp_sum_t(a.J01); a.J11 = warp_sum_t(a.J11); a.res = warp_max_t(a.res);
    if ((tid & 31) == 0) racc[tid >> 5] = a;
    __syncthreads();
    if (tid == 0) {
        RelaxAcc<T> t = racc[0];
        for (int w = 1; w < RedNT<T>::v / 32; ++w) {
            t.C0 += racc[w].C0; t.C1 += racc[w].C1; t.J00 += racc[w].J00; t.J01 += racc[w].J01;
            t.J11 += racc[w].J11; t.res = max(t.res, racc[w].res);
        }
        double *o = part + ((size_t)ridx * kRelaxBlocks + blockIdx.x) * 6;
        o[0] = t.C0; o[1] = t.C1; o[2] = t.J00; o[3] = t.J01; o[4] = t.J11; o[5] = t.res;
    }
}

// One warp per replica (one thread's chain of 64 FP64 additions per sum took 27
// us, half a sweep of two FP64 replicas' columns).
static __global__ void __launch_bounds__(128) k_g_relax_newton(const int *__restrict__ work, int nwork, RelaxIO *__restrict__ rio,
                                 const double *__restrict__ part, double tol, int iter)
{
    const int w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (w >= nwork) return;
    const int ridx = work[w];
    RelaxIO &R = rio[ridx];
    if (R.status == 0) return;
    double s[6] = {0, 0, 0, 0, 0, 0};
    for (int b = lane; b < kRelaxBlocks; b += 32) {
        const double *o = part + ((size_t)ridx * kRelaxBlocks + b) * 6;
        for (int k = 0; k < 5; ++k) s[k] += o[k];
        s[5] = fmax(s[5], o[5]);
    }
    for (int k = 0; k < 5; ++k) s[k] = warp_sum_t(s[k]);
    s[5] = warp_max_t(s[5]);
    __syncwarp();
    if (lane != 0) return;
    R.resid = s[5];
    if (s[5] < tol) {
        R.status = 0;   // converged: iters keeps the number of sweeps applied
        return;
    }
    const double det = s[2] * s[4] - s[3] * s[3];
    if (det != 0.0 && isfinite(det)) {
        R.lam[0] += -(s[4] * s[0] - s[3] * s[1]) / det;
        R.lam[1] += -(-s[3] * s[0] + s[2] * s[1]) / det;
    }
    R.iters = iter + 1;
}

template <int P, typename T>
__global__ void __launch_bounds__(CellNT<T>::v)
    k_g_relax_update(const Replica *__restrict__ reps, const int *__restrict__ work, T *__restrict__ msbase,
                     const cplx<T> *__restrict__ specbase, const RelaxIO *__restrict__ rio, double rc2_d, double eta_d)
{
    constexpr int RS = SpecGeom<P>::RS;
    const int ridx = work[blockIdx.y];
    if (rio[ridx].status == 0) return;
    const Replica &r = reps[ridx];
    const int D = r.D, DD = D * D;
    const int cell = blockIdx.x * CellNT<T>::v + threadIdx.x;
    if (cell >= DD || !r.mask[cell]) return;
    const long long ms_s = (long long)D * r.Dpad, cs = (long long)D * RS;
    const T *hr = reinterpret_cast<const T *>(specbase + r.spec_off);
    V3Ptr<T> ms{msbase + r.state_off, ms_s};
    const T relX = (T)rio[ridx].X[0], relY = (T)rio[ridx].X[1], m0 = (T)rio[ridx].lam[0], m1 = (T)rio[ridx].lam[1];
    const StepParams<T> sp = step_params<T>(r);
    const int y = cell / D, x = cell - y * D;
    const long long si = (long long)y * r.Dpad + x, hi = (long long)y * (2 * RS) + x;
    const vec3<T> b = {hr[hi] + sp.chext[0], hr[2 * cs + hi] + sp.chext[1], hr[4 * cs + hi] + sp.chext[2]};
    const T dx = (T)x - T(0.5) * (T)(D - 1) - relX, dy = (T)y - T(0.5) * (T)(D - 1) - relY;
    RelaxAcc<T> dummy = {T(0), T(0), T(0), T(0), T(0), T(0)};
    ms.st(si, relax_cell<T>(ms.ld(si), b, fm(dx, dx, dy * dy) < (T)rc2_d, dx, dy, m0, m1, (T)eta_d, dummy));
}

// The same sweep driven by an externally computed energy gradient: the field
// is b_i = gscale[r] * grad_i with gscale = -1/J (grad = dE/dm in joules, in
// the state layout), read in place of the spectrum rows.  Used by
// nd_relax_sweep_grad.
template <typename T>
__global__ void __launch_bounds__(RedNT<T>::v)
    k_relax_grad_reduce(const Replica *__restrict__ reps, const int *__restrict__ work, const T *__restrict__ mbase,
                        const T *__restrict__ gbase, const double *__restrict__ gscale,
                        const RelaxIO *__restrict__ rio, double rc2_d, double eta_d, double *__restrict__ part)
{
    __shared__ RelaxAcc<T> racc[RedNT<T>::v / 32];
    const int ridx = work[blockIdx.y], tid = threadIdx.x;
    if (rio[ridx].status == 0) return;   // CTA-uniform
    const Replica &r = reps[ridx];
    const int D = r.D, DD = D * D;
    const long long ms_s = (long long)D * r.Dpad;
    const V3Ptr<T> ms{const_cast<T *>(mbase) + r.state_off, ms_s}, gr{const_cast<T *>(gbase) + r.state_off, ms_s};
    const T relX = (T)rio[ridx].X[0], relY = (T)rio[ridx].X[1], l0 = (T)rio[ridx].lam[0], l1 = (T)rio[ridx].lam[1];
    const T eta = (T)eta_d, rc2 = (T)rc2_d, sc = (T)gscale[ridx];
    RelaxAcc<T> a = {T(0), T(0), T(0), T(0), T(0), T(0)};
    for (int cell = blockIdx.x * RedNT<T>::v + tid; cell < DD; cell += kRelaxBlocks * RedNT<T>::v) {
        if (!r.mask[cell]) continue;
        const int y = cell / D, x = cell - y * D;
        const long long si = (long long)y * r.Dpad + x;
        const vec3<T> g = gr.ld(si), b = {sc * g.x, sc * g.y, sc * g.z};
        const T dx = (T)x - T(0.5) * (T)(D - 1) - relX, dy = (T)y - T(0.5) * (T)(D - 1) - relY;
        relax_cell<T>(ms.ld(si), b, fm(dx, dx, dy * dy) < rc2, dx, dy, l0, l1, eta, a);
    }
    a.C0 = warp_sum_t(a.C0); a.C1 = warp_sum_t(a.C1); a.J00 = warp_sum_t(a.J00);
    a.J01 = warp_sum_t(a.J01); a.J11 = warp_sum_t(a.J11); a.res = warp_max_t(a.res);
    if ((tid & 31) == 0) racc[tid >> 5] = a;
    __syncthreads();
    if (tid == 0) {
        RelaxAcc<T> t = racc[0];
        for (int w = 1; w < RedNT<T>::v / 32; ++w) {
            t.C0 += racc[w].C0; t.C1 += racc[w].C1; t.J00 += racc[w].J00; t.J01 += racc[w].J01;
            t.J11 += racc[w].J11; t.res = max(t.res, racc[w].res);
        }
        double *o = part + ((size_t)ridx * kRelaxBlocks + blockIdx.x) * 6;
        o[0] = t.C0; o[1] = t.C1; o[2] = t.J00; o[3] = t.J01; o[4] = t.J11; o[5] = t.res;
    }
}

template <typename T>
__global__ void __launch_bounds__(CellNT<T>::v)
    k_relax_grad_update(const Replica *__restrict__ reps, const int *__restrict__ work, T *__restrict__ mbase,
                        const T *__restrict__ gbase, const double *__restrict__ gscale,
                        const RelaxIO *__restrict__ rio, double rc2_d, double eta_d)
{
    const int ridx = work[blockIdx.y];
    if (rio[ridx].status == 0) return;
    const Replica &r = reps[ridx];
    const int D = r.D, DD = D * D;
    const int cell = blockIdx.x * CellNT<T>::v + threadIdx.x;
    if (cell >= DD || !r.mask[cell]) return;
    const long long ms_s = (long long)D * r.Dpad;
    V3Ptr<T> ms{mbase + r.state_off, ms_s};
    const V3Ptr<T> gr{const_cast<T *>(gbase) + r.state_off, ms_s};
    const T relX = (T)rio[ridx].X[0], relY = (T)rio[ridx].X[1], m0 = (T)rio[ridx].lam[0], m1 = (T)rio[ridx].lam[1];
    const T sc = (T)gscale[ridx];
    const int y = cell / D, x = cell - y * D;
    const long long si = (long long)y * r.Dpad + x;
    const vec3<T> g = gr.ld(si), b = {sc * g.x, sc * g.y, sc * g.z};
    const T dx = (T)x - T(0.5) * (T)(D - 1) - relX, dy = (T)y - T(0.5) * (T)(D - 1) - relY;
    RelaxAcc<T> dummy = {T(0), T(0), T(0), T(0), T(0), T(0)};
    ms.st(si, relax_cell<T>(ms.ld(si), b, fm(dx, dx, dy * dy) < (T)rc2_d, dx, dy, m0, m1, (T)eta_d, dummy));
}

// One gradient-driven sweep over the replicas of one size class.
template <typename T>
static cudaError_t launch_relax_grad_t(const LaunchArgs &a, int maxD, const void *grad, const double *gscale)
{
    constexpr int NC = CellNT<T>::v, NR = RedNT<T>::v;
    const dim3 gp(kRelaxBlocks, a.nwork), gu((maxD * maxD + NC - 1) / NC, a.nwork);
    k_relax_grad_reduce<T><<<gp, NR, 0, a.stream>>>(a.reps, a.work, (const T *)a.y, (const T *)grad, gscale, a.rio,
                                                     a.rc2, a.eta, a.part);
    k_g_relax_newton<<<(a.nwork + 3) / 4, 128, 0, a.stream>>>(a.work, a.nwork, a.rio, a.part, a.tol, 0);
    k_relax_grad_update<T><<<gu, NC, 0, a.stream>>>(a.reps, a.work, (T *)a.y, (const T *)grad, gscale, a.rio, a.rc2,
                                                     a.eta);
    return cudaGetLastError();
}

// The stage buffer back to the caller's state (cells inside the disk).
template <typename T>
__global__ void k_g_store_stage(const Replica *__restrict__ reps, const int *__restrict__ work, const T *__restrict__ msbase,
                                T *__restrict__ ybase)
{
    const Replica &r = reps[work[blockIdx.y]];
    const int D = r.D, DD = D * D;
    const long long ms_s = (long long)D * r.Dpad;
    for (int cell = blockIdx.x * blockDim.x + threadIdx.x; cell < DD; cell += gridDim.x * blockDim.x) {
        if (!r.mask[cell]) continue;
        const int y = cell / D, x = cell - y * D;
        const long long si = r.state_off + (long long)y * r.Dpad + x;
        for (int c = 0; c < 3; ++c) ybase[si + c * ms_s] = msbase[si + c * ms_s];
    }
}

// --------------------------------------------------------- launch helpers


inline int fused_nt(int P, int variant)
{
    switch (P) {
    case 16: return variant == 0 ? NTV<16, 0>::v : variant == 1 ? NTV<16, 1>::v : 0;
    case 32: return variant == 0 ? NTV<32, 0>::v : variant == 1 ? NTV<32, 1>::v : 0;
    case 64: return variant == 0 ? NTV<64, 0>::v : variant == 1 ? NTV<64, 1>::v : variant == 2 ? NTV<64, 2>::v : 0;
    case 128: return variant == 0 ? NTV<128, 0>::v : variant == 1 ? NTV<128, 1>::v : 0;
    default: return 0;
    }
}
// The tiled column pass runs above P = 128 (rows of the global spectrum start
// on 32-byte sectors there).
template <int P> struct GlobTiled { static constexpr bool v = P > 128; };

template <int P, typename T, int NT>
constexpr size_t glob_smem_bytes()
{
    return sizeof(cplx<T>) *
           ((size_t)FFTGeom<P>::R1 * FFTGeom<P>::G + (size_t)groups_per_block<P, NT>() * FFTGeom<P>::SCRATCH);
}


template <int P, typename T, int MODE, int NT>
static cudaError_t launch_fused_t(const LaunchArgs &a)
{
    auto kern = k_fused<P, T, MODE, NT>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)a.smem);
    if (e != cudaSuccess) return e;
    const Segment *segs = a.segs;
    if (!segs) {
        kern<<<a.nwork, NT, a.smem, a.stream>>>(a.reps, a.work, (T *)a.y, (T *)a.acc, (T *)a.out,
                                                (const cplx<T> *)a.tw, a.nsteps, a.step_base, a.rio, a.eta, a.tol,
                                                a.rc2, a.max_iter, nullptr, nullptr, nullptr, a.wait_polls, a.status,
                                                a.use_wbuf);
        return cudaGetLastError();
    }
    // time-sliced schedule: the CTAs wait on one another, so they must all be
    // resident at once -- a cooperative launch guarantees it or fails
    const Replica *reps = a.reps;
    const int *work = a.work;
    T *y = (T *)a.y, *acc = (T *)a.acc, *out = (T *)a.out;
    const cplx<T> *tw = (const cplx<T> *)a.tw;
    long long nsteps = a.nsteps;
    unsigned long long step_base = a.step_base;
    RelaxIO *rio = a.rio;
    double eta = a.eta, tol = a.tol, rc2 = a.rc2;
    int max_iter = a.max_iter, use_wbuf = a.use_wbuf, wait_polls = a.wait_polls;
    const int *seg_off = a.seg_off;
    int *flags = a.flags;
    unsigned *status = a.status;
    void *args[] = {(void *)&reps, (void *)&work, (void *)&y, (void *)&acc, (void *)&out, (void *)&tw,
                    (void *)&nsteps, (void *)&step_base, (void *)&rio, (void *)&eta, (void *)&tol, (void *)&rc2,
                    (void *)&max_iter, (void *)&segs, (void *)&seg_off, (void *)&flags, (void *)&wait_polls,
                    (void *)&status, (void *)&use_wbuf};
    // cudaLaunchKernelEx with the cooperative attribute is also legal inside a
    // stream capture (graph kernel node)
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(a.ncta);
    cfg.blockDim = dim3(NT);
    cfg.dynamicSmemBytes = a.smem;
    cfg.stream = a.stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelExC(&cfg, (const void *)kern, args);
}

template <int P, typename T, int MODE, int NT>
static int fused_occupancy_nt(size_t smem)
{
    int n = 0;
    cudaFuncSetAttribute(k_fused<P, T, MODE, NT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_fused<P, T, MODE, NT>, NT, smem) != cudaSuccess) return 0;
    return n;
}

template <int P, typename T, int MODE>
static int fused_occupancy(int variant, size_t smem)
{
    if (variant == 1) {
        if constexpr (NTV<P, 1>::v > 0) return fused_occupancy_nt<P, T, MODE, NTV<P, 1>::v>(smem);
        return 0;
    }
    if (variant == 2) {
        if constexpr (NTV<P, 2>::v > 0) return fused_occupancy_nt<P, T, MODE, NTV<P, 2>::v>(smem);
        return 0;
    }
    return fused_occupancy_nt<P, T, MODE, NTV<P, 0>::v>(smem);
}

template <int P, typename T, int MODE>
static cudaError_t launch_stepper(const LaunchArgs &a)
{
    if (a.variant == 1) {
        if constexpr (NTV<P, 1>::v > 0) return launch_fused_t<P, T, MODE, NTV<P, 1>::v>(a);
        return cudaErrorInvalidValue;
    }
    if (a.variant == 2) {
        if constexpr (NTV<P, 2>::v > 0) return launch_fused_t<P, T, MODE, NTV<P, 2>::v>(a);
        return cudaErrorInvalidValue;
    }
    return launch_fused_t<P, T, MODE, NTV<P, 0>::v>(a);
}

template <int P, typename T>
static cudaError_t launch_fused_p(const LaunchArgs &a)
{
    constexpr int NT0 = FusedNT<P>::v;
    switch (a.mode) {
    case M_FIELD: return launch_fused_t<P, T, M_FIELD, NT0>(a);
    case M_RK4: return launch_stepper<P, T, M_RK4>(a);
    case M_HEUN: return launch_stepper<P, T, M_HEUN>(a);
    case M_RELAX: return launch_fused_t<P, T, M_RELAX, NT0>(a);
    default: return cudaErrorInvalidValue;
    }
}

template <int P, typename T, int MODE>
static void launch_g_epi(const LaunchArgs &a, dim3 ge, int stage, unsigned long long step)
{
    k_g_epi<P, T, MODE><<<ge, CellNT<T>::v, 0, a.stream>>>(a.reps, a.work, (T *)a.ms, (T *)a.y, (T *)a.acc, (T *)a.out,
                                                   (const cplx<T> *)a.spec, stage, step);
}

// Launch with programmatic stream serialisation: the kernel may be scheduled
// while its predecessor finishes, and waits for it in wait_prior_grid().
template <typename... KArgs, typename... Args>
static void launch_pdl(void (*kern)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, Args... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, kern, args...);
}

// The stepping epilogue with quad access when the state buffers allow it.
template <int P, typename T, int MODE>
static void launch_g_epi_step(const LaunchArgs &a, int maxD, int stage, unsigned long long step)
{
    const bool quad = ((reinterpret_cast<uintptr_t>(a.y) | reinterpret_cast<uintptr_t>(a.ms) |
                        reinterpret_cast<uintptr_t>(a.acc)) & 15) == 0;
    if (quad) {
        const int maxq = maxD * ((maxD + 3) / 4);
        constexpr int NC = CellNT<T>::v;
        launch_pdl(k_g_epi_quad<P, T, MODE>, dim3((maxq + NC - 1) / NC, a.nwork), dim3(NC), 0, a.stream, a.reps,
                   a.work, (T *)a.ms, (T *)a.y, (T *)a.acc, (const cplx<T> *)a.spec, stage, step);
    } else {
        launch_g_epi<P, T, MODE>(a, dim3((maxD * maxD + CellNT<T>::v - 1) / CellNT<T>::v, a.nwork), stage, step);
    }
}

// The FFT passes of one field evaluation on the global path: stage buffer ->
// spectrum (forward rows), the column pass, spectrum -> field rows in the
// spectrum buffer (inverse rows).
template <int P, typename T>
static void glob_rows(const LaunchArgs &a, int maxD, int inverse)
{
    constexpr int NT = GlobNT<T>::v, NGRP = groups_per_block<P, NT>();
    const int nrow = row_pass_tasks<P>(maxD);
    dim3 gr((nrow + NGRP - 1) / NGRP, a.nwork);
    launch_pdl(k_g_rows<P, T, NT>, gr, dim3(NT), glob_smem_bytes<P, T, NT>(), a.stream, a.reps, a.work,
               (const T *)a.ms, (cplx<T> *)a.spec, (const cplx<T> *)a.tw, inverse);
}

template <int P, typename T>
static void glob_cols(const LaunchArgs &a, int maxD)
{
    constexpr int NT = GlobNT<T>::v, NGRP = groups_per_block<P, NT>();
    if constexpr (GlobTiled<P>::v) {
        using CT = ColTile<P, T>;
        const int ntask = a.nwork * (CT::NXY + CT::NZ);
        const int grid = ntask < a.n_sm * CT::MINB ? ntask : a.n_sm * CT::MINB;
        launch_pdl(k_g_cols_tile<P, T>, dim3(grid), dim3(CT::NT), glob_smem_bytes<P, T, CT::NT>(), a.stream, a.reps,
                   a.work, a.nwork, (cplx<T> *)a.spec, (const cplx<T> *)a.tw);
    } else {
        dim3 gc((P / 2 + NGRP - 1) / NGRP, a.nwork);
        launch_pdl(k_g_cols<P, T, NT>, gc, dim3(NT), glob_smem_bytes<P, T, NT>(), a.stream, a.reps, a.work,
                   (cplx<T> *)a.spec, (const cplx<T> *)a.tw);
    }
}

template <int P, typename T>
static void glob_field_passes(const LaunchArgs &a, int maxD)
{
    glob_rows<P, T>(a, maxD, 0);
    glob_cols<P, T>(a, maxD);
    glob_rows<P, T>(a, maxD, 1);
}

// One field evaluation on the global path with its epilogue.
template <int P, typename T>
static cudaError_t glob_eval(const LaunchArgs &a, int maxD, int stage, int mode, unsigned long long step)
{
    glob_field_passes<P, T>(a, maxD);
    dim3 ge((maxD * maxD + CellNT<T>::v - 1) / CellNT<T>::v, a.nwork);
    switch (mode) {
    case M_FIELD: launch_g_epi<P, T, M_FIELD>(a, ge, stage, step); break;
    case M_RK4: launch_g_epi_step<P, T, M_RK4>(a, maxD, stage, step); break;
    case M_HEUN: launch_g_epi_step<P, T, M_HEUN>(a, maxD, stage, step); break;
    default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

template <int P, typename T>
static cudaError_t launch_global_p(const LaunchArgs &a, int maxD)
{
    constexpr int NT = GlobNT<T>::v;
    const int sm = (int)glob_smem_bytes<P, T, NT>();
    cudaError_t e0 = cudaFuncSetAttribute(k_g_rows<P, T, NT>, cudaFuncAttributeMaxDynamicSharedMemorySize, sm);
    if constexpr (!GlobTiled<P>::v) {
        if (e0 == cudaSuccess)
            e0 = cudaFuncSetAttribute(k_g_cols<P, T, NT>, cudaFuncAttributeMaxDynamicSharedMemorySize, sm);
    } else {
        if (e0 == cudaSuccess)
            e0 = cudaFuncSetAttribute(k_g_cols_tile<P, T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)glob_smem_bytes<P, T, ColTile<P, T>::NT>());
    }
    if (e0 != cudaSuccess) return e0;

    dim3 gl((maxD * maxD + 255) / 256, a.nwork);
    launch_pdl(k_g_load_stage<T>, gl, dim3(256), 0, a.stream, a.reps, a.work, (const T *)a.y, (T *)a.ms);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    if (a.mode == M_RELAX) {
        if (!a.rio || !a.part || !a.rio_host || !a.work_host) return cudaErrorInvalidValue;
        constexpr int NC = CellNT<T>::v;
        const dim3 gp(kRelaxBlocks, a.nwork), gu((maxD * maxD + NC - 1) / NC, a.nwork);
        constexpr int kCheck = 32;   // iterations between host checks for convergence of every replica
        for (int it = 0; it < a.max_iter; ++it) {
            glob_field_passes<P, T>(a, maxD);
            k_g_relax_reduce<P, T><<<gp, RedNT<T>::v, 0, a.stream>>>(a.reps, a.work, (const T *)a.ms, (const cplx<T> *)a.spec,
                                                             a.rio, a.rc2, a.eta, a.part);
            k_g_relax_newton<<<(a.nwork + 3) / 4, 128, 0, a.stream>>>(a.work, a.nwork, a.rio, a.part, a.tol, it);
            k_g_relax_update<P, T><<<gu, NC, 0, a.stream>>>(a.reps, a.work, (T *)a.ms, (const cplx<T> *)a.spec, a.rio,
                                                             a.rc2, a.eta);
            if ((e = cudaGetLastError()) != cudaSuccess) return e;
            if ((it + 1) % kCheck == 0 || it + 1 == a.max_iter) {
                // a synchronous read of the parameter array; stop once every
                // replica of this launch has converged
                if ((e = cudaMemcpyAsync(a.rio_host, a.rio, sizeof(RelaxIO) * a.n_rio, cudaMemcpyDeviceToHost,
                                         a.stream)) != cudaSuccess)
                    return e;
                if ((e = cudaStreamSynchronize(a.stream)) != cudaSuccess) return e;
                bool running = false;
                for (int k = 0; k < a.nwork && !running; ++k) running = a.rio_host[a.work_host[k]].status != 0;
                if (!running) break;
            }
        }
        k_g_store_stage<T><<<gl, 256, 0, a.stream>>>(a.reps, a.work, (const T *)a.ms, (T *)a.y);
        return cudaGetLastError();
    }
    const int nst = (a.mode == M_RK4) ? 4 : (a.mode == M_HEUN ? 2 : 1);
    const long long nsteps = a.mode == M_FIELD ? 1 : a.nsteps;
    for (long long n = 0; n < nsteps; ++n)
        for (int s = 0; s < nst; ++s) {
            e = glob_eval<P, T>(a, maxD, s, a.mode, a.step_base + n);
            if (e != cudaSuccess) return e;
        }
    return cudaSuccess;
}

}  // namespace nd
