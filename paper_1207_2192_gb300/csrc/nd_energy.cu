// nd_energy.cu -- the energy of Eq. Hmm and its thickness derivative in FP64.
//
// Both are quadratic forms of the state in the spectral kernel, so they need
// the forward transforms only (Parseval): with X, Y, Z the P x P transforms of
// the masked components and G the kernel that holds the exchange and 1/P^2,
//   E/J = -1/2 sum_k [G_xx |X|^2 + G_yy |Y|^2 + G_zz |Z|^2 + 2 G_xy Re(X Y*)] - c h_ext . M(0),
// and the same sum with the derivative kernel gives d(E/J)/dl.  GB300 issues an
// FP64 instruction per SM sub-partition every 64 to 76 cycles whatever the
// number of active lanes, so what counts is the number of warp instructions
// and that all sub-partitions have a warp:
//   k_energy_rows  one FFT group per row task, small CTAs over all replicas;
//   k_energy_cols  three groups per column slot (x, y, z), each transforms its
//                  column and sums its part of both forms; the last CTA of a
//                  replica adds the partial sums in a fixed order.
// Sixteen replicas of R = 60 nm (P = 128), energies with dE/dL, cold cache: the
// former two field evaluations (rows, columns there and back, epilogue) took
// 2 x 240 us; the rows here take 18 us (21 in CTAs of four warps), the columns 47.
#include <math.h>

#include "nd_phases.cuh"
#include "nd_kernels.h"

namespace nd {

// A row of the state as the transforms read it: zero outside the disk.
template <typename S> struct MaskedRow {
    const S *p;
    const unsigned char *mask;
    __device__ __forceinline__ double operator[](int x) const { return mask[x] ? (double)p[x] : 0.0; }
};

constexpr int kRowThreads = 32;   // one warp: the row tasks spread over every sub-partition

template <int P, typename S>
__global__ void __launch_bounds__(kRowThreads)
    k_energy_rows(const Replica *__restrict__ reps, const int *__restrict__ work, const S *__restrict__ mbase,
                  cplx<double> *__restrict__ specbase, long long spec_stride, const cplx<double> *__restrict__ twP)
{
    using Gm = FFTGeom<P>;
    constexpr int G = Gm::G, R1 = Gm::R1, RS = SpecGeom<P>::RS, NGRP = groups_per_block<P, kRowThreads>();
    extern __shared__ __align__(16) unsigned char esm[];
    cplx<double> *tw = reinterpret_cast<cplx<double> *>(esm), *scratch = tw + R1 * G;
    load_twiddles<P>(tw, twP, threadIdx.x, kRowThreads);
    const Replica &r = reps[work[blockIdx.y]];
    const int D = r.D, nrow = row_pass_tasks<P>(D);
    __syncthreads();
    GroupId<P> gid(threadIdx.x);
    if (!gid.valid) return;
    const int q = blockIdx.x * NGRP + gid.group;
    const bool act = q < nrow;
    const long long cs = (long long)D * RS, ms = (long long)D * r.Dpad;
    cplx<double> *spec = specbase + (spec_stride ? blockIdx.y * spec_stride : r.spec_off), *scr = scratch + gid.group * Gm::SCRATCH;
    auto row = [&](int c, int y) {
        return MaskedRow<S>{mbase + r.state_off + c * ms + (long long)y * r.Dpad, r.mask + (long long)y * D};
    };
    if constexpr (HalfRows<P>::on) {
        const int c = act ? q / D : 0, y = act ? q - c * D : 0;
        row_fwd_half<P, double>(act, row(c, y), D, spec + c * cs + (long long)y * RS, gid.t, scr, tw, gid.gmask);
    } else {
        const bool isxy = q < D;
        const int y0 = !act ? 0 : isxy ? q : 2 * (q - D), y1 = y0 + 1;
        const bool hasB = act && (isxy || y1 < D);
        const int cA = isxy ? 0 : 2, cB = isxy ? 1 : 2, yB = isxy ? y0 : y1;
        const MaskedRow<S> a = row(cA, y0), b = row(cB, hasB ? yB : y0);
        cplx<double> v[R1];
#pragma unroll
        for (int o = 0; o < R1; ++o) {
            const int x = gid.t + G * o;
            v[o] = {act && o < R1 / 2 && x < D ? a[x] : 0.0, hasB && o < R1 / 2 && x < D ? b[x] : 0.0};
        }
        row_fwd_core<P, double>(v, act, spec + cA * cs + (long long)y0 * RS, spec + cB * cs + (long long)yB * RS, hasB,
                                gid.t, scr, tw, gid.gmask);
    }
}

// Three warps: with G a power of two, warp c holds component c of 32/G slots;
// with ten-lane groups each warp holds the three components of one slot.
template <int P> struct EnergyCols {
    static constexpr int NT = 96;
    static constexpr bool POW2 = FFTGeom<P>::POW2;
    static constexpr int SLOTS = POW2 ? 32 / FFTGeom<P>::G : 3;
    static constexpr int NBLK = (P / 2 + SLOTS - 1) / SLOTS;
};

template <int P>
__global__ void __launch_bounds__(96)
    k_energy_cols(const Replica *__restrict__ reps, const int *__restrict__ work, const cplx<double> *__restrict__ specbase,
                  long long spec_stride, const cplx<double> *__restrict__ twP, double *__restrict__ part, unsigned *__restrict__ done,
                  double *__restrict__ out, int with_dl)
{
    using Gm = FFTGeom<P>;
    using EC = EnergyCols<P>;
    constexpr int G = Gm::G, R1 = Gm::R1, RS = SpecGeom<P>::RS, KH = SpecGeom<P>::KH, KK = KH * KH;
    extern __shared__ __align__(16) unsigned char esm[];
    __shared__ double red[3][2];
    __shared__ bool last_s;
    cplx<double> *tw = reinterpret_cast<cplx<double> *>(esm), *scratch = tw + R1 * G;
    const int tid = threadIdx.x, warp = tid >> 5;
    load_twiddles<P>(tw, twP, tid, EC::NT);
    const int ridx = work[blockIdx.y];
    const Replica &r = reps[ridx];
    const int D = r.D;
    __syncthreads();
    GroupId<P> gid(tid);
    const int gw = gid.valid ? gid.group - warp * Gm::GROUPS_PER_WARP : 0;   // group of the warp
    const int c = EC::POW2 ? warp : gw, slot = EC::POW2 ? gw : warp;
    const int q = blockIdx.x * EC::SLOTS + slot;   // column slot: kx = q, slot 0 the packed pair kx = 0, P/2
    const bool act = gid.valid && q < P / 2, packed = q == 0;
    cplx<double> *scr = scratch + gid.group * Gm::SCRATCH;
    const cplx<double> *scry = scratch + (EC::POW2 ? 1 * Gm::GROUPS_PER_WARP + slot : warp * Gm::GROUPS_PER_WARP + 1) * Gm::SCRATCH;
    double e = 0.0, el = 0.0;
    cplx<double> v[R1];
    if (gid.valid) {
        const cplx<double> *col = specbase + (spec_stride ? blockIdx.y * spec_stride : r.spec_off) + c * (long long)D * RS;
        col_load_kind<P, double>(v, const_cast<cplx<double> *>(col), packed, act ? q : 1, D, gid.t, act);
        fft_group<P, -1, FFT_HALF_IN>(v, gid.t, scr, tw, gid.gmask);
        mirror_put<P>(v, scr, gid.t);   // natural order: the packed pair's mirror, the x groups' y spectra
    }
    __syncthreads();
    if (act) {
        const double *g64 = r.Ghat64 + 4 * KK, *gl = r.GhatL + 4 * KK;   // component-major
        const int comp = c == 2 ? 3 : c;                                 // the diagonal entry
#pragma unroll
        for (int o = 0; o < R1; ++o) {
            const int ky = gid.t + G * o;
            const bool up = ky <= P / 2;
            const int kyr = up ? ky : P - ky;
            const int i = comp * KK + q * KH + kyr, i2 = comp * KK + (P / 2) * KH + kyr, ix = 2 * KK + q * KH + kyr;
            if (packed) {   // the spectra of the two real columns, once each (G_xy vanishes there)
                const cplx<double> w = mirror_get<P>(scr, ky);
                const cplx<double> F0 = {0.5 * (v[o].x + w.x), 0.5 * (v[o].y - w.y)};
                const cplx<double> F1 = {0.5 * (v[o].y + w.y), -0.5 * (v[o].x - w.x)};
                const double p0 = 0.5 * fm(F0.x, F0.x, F0.y * F0.y), p1 = 0.5 * fm(F1.x, F1.x, F1.y * F1.y);
                e = fm(__ldg(g64 + i), p0, fm(__ldg(g64 + i2), p1, e));
                if (with_dl) el = fm(__ldg(gl + i), p0, fm(__ldg(gl + i2), p1, el));
                if (ky == 0) e = fm(r.chext[c], F0.x, e);
            } else {        // k and its conjugate at P - kx: twice the half
                const double p = fm(v[o].x, v[o].x, v[o].y * v[o].y);
                e = fm(__ldg(g64 + i), p, e);
                if (with_dl) el = fm(__ldg(gl + i), p, el);
                if (c == 0) {
                    const cplx<double> y = scry[ky];
                    const double re = 2.0 * fm(v[o].x, y.x, v[o].y * y.y), s = up ? re : -re;   // G_xy is odd in ky
                    e = fm(__ldg(g64 + ix), s, e);
                    if (with_dl) el = fm(__ldg(gl + ix), s, el);
                }
            }
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        e += __shfl_xor_sync(0xffffffffu, e, o);
        el += __shfl_xor_sync(0xffffffffu, el, o);
    }
    if ((tid & 31) == 0) { red[warp][0] = e; red[warp][1] = el; }
    __syncthreads();
    double *pr = part + (size_t)ridx * 2 * EC::NBLK;
    if (tid == 0) {
        __stcg(pr + 2 * blockIdx.x, red[0][0] + red[1][0] + red[2][0]);
        __stcg(pr + 2 * blockIdx.x + 1, red[0][1] + red[1][1] + red[2][1]);
        __threadfence();
        last_s = atomicInc(done + ridx, EC::NBLK - 1) == EC::NBLK - 1;   // (wraps to zero for the next call)
    }
    __syncthreads();
    if (last_s && tid < 32) {
        __threadfence();
        double s = 0.0, sl = 0.0;
        for (int b = tid; b < EC::NBLK; b += 32) {
            s += __ldcg(pr + 2 * b);
            sl += __ldcg(pr + 2 * b + 1);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            s += __shfl_xor_sync(0xffffffffu, s, o);
            sl += __shfl_xor_sync(0xffffffffu, sl, o);
        }
        if (tid == 0) {
            out[2 * ridx] = -s;
            out[2 * ridx + 1] = -sl;
        }
    }
}

template <int P, typename S>
static cudaError_t launch_p(const EnergyArgs &a)
{
    constexpr int NGRP = groups_per_block<P, kRowThreads>();
    constexpr size_t tab = sizeof(cplx<double>) * FFTGeom<P>::R1 * FFTGeom<P>::G;
    constexpr size_t sr = tab + sizeof(cplx<double>) * (size_t)NGRP * FFTGeom<P>::SCRATCH;
    constexpr size_t sc = tab + sizeof(cplx<double>) * (size_t)3 * FFTGeom<P>::GROUPS_PER_WARP * FFTGeom<P>::SCRATCH;
    cudaError_t e = cudaFuncSetAttribute(k_energy_rows<P, S>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sr);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_energy_cols<P>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sc);
    if (e != cudaSuccess) return e;
    k_energy_rows<P, S><<<dim3((row_pass_tasks<P>(a.maxD) + NGRP - 1) / NGRP, a.nwork), kRowThreads, sr, a.stream>>>(
        a.reps, a.work, (const S *)a.m, (cplx<double> *)a.spec, a.spec_stride, (const cplx<double> *)a.tw);
    k_energy_cols<P><<<dim3(EnergyCols<P>::NBLK, a.nwork), EnergyCols<P>::NT, sc, a.stream>>>(
        a.reps, a.work, (const cplx<double> *)a.spec, a.spec_stride, (const cplx<double> *)a.tw, a.part, a.done, a.out, a.with_dl);
    return cudaGetLastError();
}

cudaError_t launch_energy(int P, int prec, const EnergyArgs &a)
{
    switch (P) {
#define X(p) case p: return prec == ND_PREC_FP64 ? launch_p<p, double>(a) : launch_p<p, float>(a);
    X(16) X(32) X(64) X(128) X(192) X(200) X(256) X(512) X(1024)
#undef X
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace nd
