// nd_aux.cu -- once-per-geometry spectral kernel build and the small
// per-replica kernels: analytic vortex profile, vortex-core estimator, <m>,
// finiteness scan.
#include <math.h>

#include "nd_common.cuh"
#include "nd_kernels.h"
#include "nd_schedule.h"

namespace nd {

// --------------------------------------------------- spectral kernel build

// a^2 G at cell displacement (dx, dy) >= 0, lengths in units of a (Section
// II.B): G_zz = -l/(2 pi r s (s+r)), G_xx = l/(2 pi r^4) (x^2/s - y^2/(s+r)),
// G_xy = l/(2 pi r^4) (2s+r)/(s+r) x y/s, s = sqrt(r^2 + l^2); the origin holds
// the cell self terms -Nx, -Nx, 0, -Nz.
__global__ void k_green_quarter(int D, double l, double Nx, double Nz, double *Gq)
{
    const int n = D * D;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const int dy = i / D, dx = i - dy * D;
        double xx, yy, xy, zz;
        if (dx == 0 && dy == 0) {
            xx = -Nx; yy = -Nx; xy = 0.0; zz = -Nz;
        } else {
            const double x = dx, y = dy, r2 = x * x + y * y, r = sqrt(r2), s = sqrt(r2 + l * l);
            const double pre = l / (2.0 * M_PI * r2 * r2);
            xx = pre * (x * x / s - y * y / (s + r));
            yy = pre * (y * y / s - x * x / (s + r));
            xy = pre * ((2.0 * s + r) / (s + r)) * (x * y / s);
            zz = -l / (2.0 * M_PI * r * s * (s + r));
        }
        Gq[i] = xx; Gq[n + i] = yy; Gq[2 * n + i] = xy; Gq[3 * n + i] = zz;
    }
}

// Thickness derivative of the table above, d(a^2 G)/dl at fixed displacement
// (lengths in units of a), and of the self terms:
//   dN_z/dl = r_o (r_o - q)/(q l^2),  dN_x/dl = r_o (q - r_o)/(2 q l^2),  q = sqrt(l^2 + r_o^2).
__global__ void k_green_quarter_dl(int D, double l, double dNx, double dNz, double *Gq)
{
    const int n = D * D;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const int dy = i / D, dx = i - dy * D;
        double xx, yy, xy, zz;
        if (dx == 0 && dy == 0) {
            xx = -dNx; yy = -dNx; xy = 0.0; zz = -dNz;
        } else {
            const double x = dx, y = dy, r2 = x * x + y * y, r = sqrt(r2), s = sqrt(r2 + l * l);
            const double ds = l / s, r4 = r2 * r2;
            // G_xx = l/(2 pi r^4) (x^2/s - y^2/(s+r))
            xx = (1.0 / (2.0 * M_PI * r4)) * ((x * x / s - y * y / (s + r)) + l * (-x * x * ds / (s * s) + y * y * ds / ((s + r) * (s + r))));
            yy = (1.0 / (2.0 * M_PI * r4)) * ((y * y / s - x * x / (s + r)) + l * (-y * y * ds / (s * s) + x * x * ds / ((s + r) * (s + r))));
            // G_xy = g(l) x y / (2 pi r^4), g = l (2s+r)/((s+r) s)
            const double den = (s + r) * s;
            const double g = (2.0 * s + r) / den + l * ds * (2.0 * (s + r) * s - (2.0 * s + r) * (2.0 * s + r)) / (den * den);
            xy = g * x * y / (2.0 * M_PI * r4);
            // G_zz = -f(l)/(2 pi r), f = l/(s (s+r))
            const double f = (s * (s + r) - l * ds * (2.0 * s + r)) / (den * den);
            zz = -f / (2.0 * M_PI * r);
        }
        Gq[i] = xx; Gq[n + i] = yy; Gq[2 * n + i] = xy; Gq[3 * n + i] = zz;
    }
}

__global__ void k_trig_table(int P, double *cs)
{
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < P; k += gridDim.x * blockDim.x) {
        double s, c;
        sincospi(2.0 * k / P, &s, &c);
        cs[2 * k] = c; cs[2 * k + 1] = s;
    }
}

// Pass 1 over dx: T1[c][dy][kx] = sum_dx w(dx) Gq[c][dy][dx] f_c(2 pi kx dx / P),
// f = cos for the even components (xx, yy, zz), sin for the odd one (xy),
// w = 1 at dx = 0 and 2 otherwise (the two signs of dx folded together).
__global__ void k_ghat_pass1(int P, int D, const double *Gq, const double *cs, double *T1)
{
    const int KH = P / 2 + 1, n = 4 * D * KH;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const int kx = i % KH, dy = (i / KH) % D, c = i / (KH * D);
        const double *g = Gq + (size_t)c * D * D + (size_t)dy * D;
        const double *fc = cs + (c == 2 ? 1 : 0);
        double acc = g[0] * fc[0];
        // phase index kx*dx mod P, advanced by kx per term
        for (int dx = 1, k = kx; dx < D; ++dx, k = (k + kx >= P) ? k + kx - P : k + kx) acc += 2.0 * g[dx] * fc[2 * k];
        T1[i] = acc;
    }
}

// Pass 2 over dy and final assembly into [kx][ky][4], followed by the same
// values component-major, [4][kx][ky]:
//   Ghat_c = s_c sum_dy w(dy) T1[c][dy][kx] f_c(2 pi ky dy / P), s_xy = -1,
//   diagonal: (c Ghat + 2 cos(2 pi kx/P) + 2 cos(2 pi ky/P)) / P^2 (exchange folded in),
//   xy:       c Ghat_xy / P^2.
__global__ void k_ghat_pass2(int P, int D, double cfac, const double *T1, const double *cs, double *G64, float *G32,
                             int with_exchange)
{
    const int KH = P / 2 + 1, n = KH * KH;
    const double inv = 1.0 / ((double)P * (double)P);
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const int kx = i / KH, ky = i % KH;
        double v[4];
        for (int c = 0; c < 4; ++c) {
            const double *t1 = T1 + (size_t)c * D * KH + kx;
            const double *fc = cs + (c == 2 ? 1 : 0);
            double acc = t1[0] * fc[0];
            for (int dy = 1, k = ky; dy < D; ++dy, k = (k + ky >= P) ? k + ky - P : k + ky)
                acc += 2.0 * t1[(size_t)dy * KH] * fc[2 * k];
            v[c] = (c == 2) ? -acc : acc;
        }
        const double kex = with_exchange ? 2.0 * cs[2 * kx] + 2.0 * cs[2 * ky] : 0.0;
        const double o[4] = {(cfac * v[0] + kex) * inv, (cfac * v[1] + kex) * inv, cfac * v[2] * inv,
                             (cfac * v[3] + kex) * inv};
        for (int c = 0; c < 4; ++c) {
            G64[(size_t)i * 4 + c] = o[c];
            if (G32) G32[(size_t)i * 4 + c] = (float)o[c];
            // the same values component-major after the interleaved block
            G64[(size_t)(4 + c) * n + i] = o[c];
            if (G32) G32[(size_t)(4 + c) * n + i] = (float)o[c];
        }
    }
}

size_t build_ghat_work_doubles(int P, int D) { return (size_t)4 * D * D + (size_t)4 * D * (P / 2 + 1) + 2 * (size_t)P; }

cudaError_t build_ghat(int P, int D, double l, double Nx, double Nz, double cfac, const double *Gq_dev, double *G64,
                       float *G32, double *work, cudaStream_t st)
{
    double *Gq = work, *T1 = Gq + (size_t)4 * D * D, *cs = T1 + (size_t)4 * D * (P / 2 + 1);
    if (Gq_dev) {
        cudaError_t e = cudaMemcpyAsync(Gq, Gq_dev, sizeof(double) * 4 * D * D, cudaMemcpyDeviceToDevice, st);
        if (e != cudaSuccess) return e;
    } else {
        k_green_quarter<<<(D * D + 255) / 256, 256, 0, st>>>(D, l, Nx, Nz, Gq);
    }
    k_trig_table<<<(P + 255) / 256, 256, 0, st>>>(P, cs);
    const int KH = P / 2 + 1;
    k_ghat_pass1<<<(4 * D * KH + 255) / 256, 256, 0, st>>>(P, D, Gq, cs, T1);
    k_ghat_pass2<<<(KH * KH + 127) / 128, 128, 0, st>>>(P, D, cfac, T1, cs, G64, G32, 1);
    return cudaGetLastError();
}

cudaError_t build_ghat_dl(int P, int D, double l, double dNx, double dNz, double cfac, double *GL64, double *work,
                          cudaStream_t st)
{
    double *Gq = work, *T1 = Gq + (size_t)4 * D * D, *cs = T1 + (size_t)4 * D * (P / 2 + 1);
    k_green_quarter_dl<<<(D * D + 255) / 256, 256, 0, st>>>(D, l, dNx, dNz, Gq);
    k_trig_table<<<(P + 255) / 256, 256, 0, st>>>(P, cs);
    const int KH = P / 2 + 1;
    k_ghat_pass1<<<(4 * D * KH + 255) / 256, 256, 0, st>>>(P, D, Gq, cs, T1);
    k_ghat_pass2<<<(KH * KH + 127) / 128, 128, 0, st>>>(P, D, cfac, T1, cs, GL64, nullptr, 0);
    return cudaGetLastError();
}

// -------------------------------------------------------- vortex profile

// Planar q = +1 vortex at X0 (Section IV) with a seeded core:
// phi = atan2(y - y0, x - x0) + chirality pi/2, m_z = polarity exp(-rho^2/lambda^2).
template <typename T>
__global__ void k_init_vortex(const Replica *reps, const int *work, T *ybase, const double *X0, const int *pc,
                              double lam)
{
    const int ridx = work[blockIdx.y];
    const Replica r = reps[ridx];
    const int D = r.D, DD = D * D;
    const long long cs = (long long)D * r.Dpad;
    const double x0 = X0[2 * ridx], y0 = X0[2 * ridx + 1];
    const int pol = pc[2 * ridx], chi = pc[2 * ridx + 1];
    T *y = ybase + r.state_off;
    for (int cell = blockIdx.x * blockDim.x + threadIdx.x; cell < DD; cell += gridDim.x * blockDim.x) {
        const int j = cell / D, i = cell - j * D;
        const long long si = (long long)j * r.Dpad + i;
        double mx = 0, my = 0, mz = 0;
        if (r.mask[cell]) {
            const double x = i - 0.5 * (D - 1), yy = j - 0.5 * (D - 1);
            const double rho2 = (x - x0) * (x - x0) + (yy - y0) * (yy - y0);
            mz = pol * exp(-rho2 / (lam * lam));
            const double phi = atan2(yy - y0, x - x0) + chi * 0.5 * M_PI;
            const double sp = sqrt(1.0 - mz * mz);
            double sn, cn;
            sincos(phi, &sn, &cn);
            mx = sp * cn; my = sp * sn;
        }
        y[si] = (T)mx; y[cs + si] = (T)my; y[2 * cs + si] = (T)mz;
    }
    // cells of the padded columns stay untouched
}

cudaError_t launch_init_vortex(int prec, const Replica *reps, const int *work, int nwork, int maxD, void *y,
                               const double *X0, const int *pc, double lam, cudaStream_t st)
{
    dim3 g((maxD * maxD + 255) / 256, nwork);
    if (prec == ND_PREC_FP64) k_init_vortex<double><<<g, 256, 0, st>>>(reps, work, (double *)y, X0, pc, lam);
    else k_init_vortex<float><<<g, 256, 0, st>>>(reps, work, (float *)y, X0, pc, lam);
    return cudaGetLastError();
}

// ------------------------------------------------------------ vortex core

// Core position estimator (Section IV) in one kernel: grid (nblk, replicas),
// each CTA stages a strip of rows of the in-plane components in shared memory
// (one batch of loads instead of a chain per plaquette) and scans its plaquettes
// for the winding +1 one with the largest m_z^2 corner sum (lowest index on
// ties), and the last CTA of a replica picks the best candidate (same rule) and forms the m_z^2-weighted
// centroid over the disk cells within 4 lambda_ex of it, visiting only the
// bounding box of that circle.  The winding and the corner sums are those of
// double precision with no fused multiply-adds, in the same order as the CPU
// reference, so both take the same integer decisions from the same inputs; but
// FP64 issues one warp instruction per 64-76 cycles here, so the scan reads the
// winding off the signs (below) and only single plaquettes reach FP64.  256
// replicas of D = 50, cold cache: 23.6 + 15.4 us as two kernels with an
// arctangent per corner and FP64 trees over the CTA, 19.9 us now.
template <typename T> struct CoreAt {
    const T *y;
    long long cs;
    int D, Dpad;
    __device__ __forceinline__ double operator()(int cell, int c) const { return (double)raw(cell, c); }
    __device__ __forceinline__ T raw(int cell, int c) const
    {
        const int j = cell / D, i = cell - j * D;
        return y[c * cs + (long long)j * Dpad + i];
    }
};

// Winding of the plaquette with corners c[0..3] in counter-clockwise order: the
// sum over its edges of the turn in (-pi, pi], over 2 pi.  An edge adds a
// revolution to the difference of the corners' polar angles exactly where it
// crosses the negative x axis the short way: from y >= 0 to y < 0 turning
// left, or back turning right.  The signs of the cross products decide that;
// where one that matters is within rounding of zero (the corners antiparallel),
// or a corner's in-plane part is too small for single-precision products, the
// turns are summed in double precision.
template <typename T>
__device__ __forceinline__ int winding(const CoreAt<T> &at, const int (&c)[4], const float (&px)[4],
                                       const float (&py)[4])
{
    bool sure = true;
    for (int q = 0; q < 4; ++q)
        sure &= px[q] * px[q] + py[q] * py[q] > 1e-12f && fabsf(py[q]) > 1e-30f;
    int w = 0;
    for (int q = 0; q < 4; ++q) {
        const int n = (q + 1) & 3;
        if ((py[q] < 0.0f) == (py[n] < 0.0f)) continue;
        const float u = px[q] * py[n], v = py[q] * px[n], cr = u - v;
        sure &= fabsf(cr) > 1e-5f * (fabsf(u) + fabsf(v));
        if (py[q] >= 0.0f && cr > 0.0f) ++w;
        if (py[q] < 0.0f && cr < 0.0f) --w;
    }
    if (sure) return w;
    double s = 0.0;
    for (int q = 0; q < 4; ++q) {
        const int p0 = c[q], p1 = c[(q + 1) & 3];
        const double ax = at(p0, 0), ay = at(p0, 1), bx = at(p1, 0), by = at(p1, 1);
        const double cr = __dsub_rn(__dmul_rn(ax, by), __dmul_rn(ay, bx));
        const double dt = __dadd_rn(__dmul_rn(ax, bx), __dmul_rn(ay, by));
        s = __dadd_rn(s, atan2(cr, dt));
    }
    return (int)llround(s / (2.0 * M_PI));
}

// A candidate plaquette: corner sum (negative: none) and index.
struct CoreCand {
    double w;
    int i;
    __device__ __forceinline__ void take(double w2, int i2)
    {
        if (w2 > w || (w2 == w && i2 < i)) { w = w2; i = i2; }
    }
};

// The circle of radius rc' = sqrt(rc2) around the plaquette's centre: the half
// side of its bounding box, and (2 dx)^2 + (2 dy)^2 < n4 (odd integers) for
// dx^2 + dy^2 < rc2.
struct CoreBox {
    int rc;
    long long n4;
};

template <typename T>
__global__ void __launch_bounds__(256) k_core(const Replica *reps, const int *work, const T *ybase, double *part,
                                              unsigned *done, CoreBox box, double *out)
{
    extern __shared__ __align__(16) float strip[];
    __shared__ CoreCand wc[8];
    __shared__ CoreCand best_s;
    __shared__ double sx[3][4];
    __shared__ bool last_s;
    const int ridx = work[blockIdx.y], nblk = gridDim.x;
    const Replica &r = reps[ridx];
    const int D = r.D, tid = threadIdx.x;
    const unsigned char *mask = r.mask;
    const CoreAt<T> at{ybase + r.state_off, (long long)D * r.Dpad, D, r.Dpad};
    CoreCand cand = {-1.0, 0x7fffffff};
    // rows ja..jb of the strip's plaquettes, the row after the last included;
    // cells outside the disk are marked with a NaN
    const int H = (D - 1 + nblk - 1) / nblk, ja = min(blockIdx.x * H, D - 1), jb = min(ja + H, D - 1);
    float2 *const sp = reinterpret_cast<float2 *>(strip);
    const T *y0 = ybase + r.state_off;
    const int ncell = (jb - ja + 1) * D;
#pragma unroll 4
    for (int k = tid; k < ncell; k += 256) {
        const int jr = k / D, i = k - jr * D;
        const long long si = (long long)(ja + jr) * r.Dpad + i;
        const float x = (float)y0[si], y = (float)y0[at.cs + si];
        sp[k] = make_float2(mask[ja * D + k] ? x : __int_as_float(0x7fffffff), y);
    }
    __syncthreads();
    const int np = (jb - ja) * (D - 1);
    for (int p = tid; p < np; p += 256) {
        const int jr = p / (D - 1), i = p - jr * (D - 1), k = jr * D + i;
        const int t = ja * D + k;
        const float2 q0 = sp[k], q1 = sp[k + 1], q2 = sp[k + D + 1], q3 = sp[k + D];
        const int c[4] = {t, t + 1, t + D + 1, t + D};
        const float px[4] = {q0.x, q1.x, q2.x, q3.x}, py[4] = {q0.y, q1.y, q2.y, q3.y};
        if (!(px[0] == px[0] && px[1] == px[1] && px[2] == px[2] && px[3] == px[3])) continue;
        if (winding(at, c, px, py) != 1) continue;
        const double z0 = at(t, 2), z1 = at(t + 1, 2), z2 = at(t + D, 2), z3 = at(t + D + 1, 2);
        double w = __dmul_rn(z0, z0);
        w = __dadd_rn(w, __dmul_rn(z1, z1));
        w = __dadd_rn(w, __dmul_rn(z2, z2));
        w = __dadd_rn(w, __dmul_rn(z3, z3));
        cand.take(w, t);
    }
    // candidates are rare: a warp compares only the lanes that hold one
    CoreCand b = {-1.0, 0x7fffffff};
    for (unsigned m = __ballot_sync(0xffffffffu, cand.i != 0x7fffffff); m; m &= m - 1) {
        const int l = __ffs(m) - 1;
        b.take(__shfl_sync(0xffffffffu, cand.w, l), __shfl_sync(0xffffffffu, cand.i, l));
    }
    if ((tid & 31) == 0) wc[tid >> 5] = b;
    __syncthreads();
    if (tid == 0) {
        for (int k = 1; k < 8; ++k)
            if (wc[k].i != 0x7fffffff) wc[0].take(wc[k].w, wc[k].i);
        best_s = wc[0];
        last_s = true;
        if (nblk > 1) {
            double *o = part + 2 * ((size_t)ridx * nblk + blockIdx.x);
            __stcg(o, best_s.w);
            __stcg(o + 1, (double)best_s.i);
            __threadfence();
            last_s = atomicInc(done + ridx, nblk - 1) == nblk - 1;   // (wraps to zero for the next call)
            if (last_s) {
                __threadfence();
                CoreCand g = {-1.0, 0x7fffffff};
                for (int k = 0; k < nblk; ++k) {
                    const double w = __ldcg(part + 2 * ((size_t)ridx * nblk + k));
                    if (w >= 0.0) g.take(w, (int)__ldcg(part + 2 * ((size_t)ridx * nblk + k) + 1));
                }
                best_s = g;
            }
        }
    }
    __syncthreads();
    if (!last_s) return;
    const int best = best_s.i;
    const bool found = best != 0x7fffffff;
    // Four warps, one per sub-partition.  Bound by FP64 issue: five
    // instructions a cell (the conversions by bits), six additions a warp.
    double a0 = 0, a1 = 0, a2 = 0;
    if (tid < 128) {
        if (found) {
            const int bj = best / D, bii = best - bj * D;
            const int i0 = max(0, bii - box.rc), i1 = min(D - 1, bii + 1 + box.rc);
            const int j0 = max(0, bj - box.rc), j1 = min(D - 1, bj + 1 + box.rc);
            const int w = i1 - i0 + 1, nbox = w * (j1 - j0 + 1);
#pragma unroll 4
            for (int k = tid; k < nbox; k += 128) {
                const int jr = k / w, j = j0 + jr, i = i0 + k - jr * w, cell = j * D + i;
                const int ex = 2 * (i - bii) - 1, ey = 2 * (j - bj) - 1;
                const bool in = (long long)ex * ex + (long long)ey * ey < box.n4 && mask[cell];
                const T zt = at.raw(cell, 2);
                if (!in) continue;
                const double z = to_double(zt), wz = z * z;
                // twice the coordinates from the grid's centre are integers
                a0 += wz;
                a1 += wz * to_double((float)(2 * i - (D - 1)));
                a2 += wz * to_double((float)(2 * j - (D - 1)));
            }
        }
        const double s = warp_sum3(a0, a1, a2);
        if ((tid & 7) == 0 && (tid & 31) < 24) sx[(tid & 31) >> 3][tid >> 5] = s;
    }
    __syncthreads();
    if (tid < 32) {   // lanes 4c..4c+3 sum component c's four warps
        double v = tid < 12 ? sx[tid >> 2][tid & 3] : 0.0;
        for (int o = 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        const double w = __shfl_sync(0xffffffffu, v, 0);
        const bool ok = found && w > 0.0;
        double *o = out + 4 * ridx;
        if (tid == 4 || tid == 8) o[(tid >> 2) - 1] = ok ? 0.5 * v / w : 0.0;
        if (tid == 0) {
            o[2] = ok ? 0.0 : 1.0;
            o[3] = found ? (double)best : -1.0;
        }
    }
}

// CTAs of a replica's scan: strips of about 4096 cells (a 33 KB stage), at
// most kCoreMaxBlocks.
static int core_scan_blocks(int D)
{
    const int n = (D * D + 4095) / 4096;
    return n > kCoreMaxBlocks ? kCoreMaxBlocks : n;
}

cudaError_t launch_vortex_core(int prec, const Replica *reps, const int *work, int nwork, int maxD, const void *y,
                               double rc2, double *part, unsigned *done, double *out, cudaStream_t st)
{
    const int nblk = core_scan_blocks(maxD);
    const dim3 g(nblk, nwork);
    const CoreBox box = {(int)ceil(sqrt(rc2)) + 1, (long long)ceil(4.0 * rc2)};
    const size_t sm = sizeof(float2) * ((size_t)(maxD - 1 + nblk - 1) / nblk + 1) * maxD;   // <= 41 KB
    if (prec == ND_PREC_FP64) k_core<double><<<g, 256, sm, st>>>(reps, work, (const double *)y, part, done, box, out);
    else k_core<float><<<g, 256, sm, st>>>(reps, work, (const float *)y, part, done, box, out);
    return cudaGetLastError();
}

// Advance the noise-step counter of every replica (graph replays continue the
// Philox stream where the previous replay stopped).
__global__ void k_advance_steps(Replica *reps, int n, long long steps)
{
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r < n) reps[r].step0 += (unsigned long long)steps;
}

cudaError_t launch_advance_steps(Replica *reps, int n, long long steps, cudaStream_t s)
{
    k_advance_steps<<<(n + 127) / 128, 128, 0, s>>>(reps, n, steps);
    return cudaGetLastError();
}

// ------------------------------------------------------------ statistics

// Per-replica accumulation of the core statistics of Sec. V.C in double
// precision with 64-bit histogram counts: samples where a vortex was found
// add r = |r_c| to <x>, <y>, <r^2> and to the r histogram; consecutive found
// samples add the speed V = |r_c(t) - r_c(t - dt)|/dt to <V^2> and the V
// histogram.  One thread per replica; core holds the estimator output in
// cell units ([4] per replica: x, y, status, plaquette).
__global__ void k_stats_update(const int *work, int nwork, const double *core, const double *a_of_rep,
                               StatsAcc *st, unsigned long long *hr, unsigned long long *hv, int rb, int vb,
                               double r_max, double v_max, double dt)
{
    const int w = blockIdx.x * blockDim.x + threadIdx.x;
    if (w >= nwork) return;
    const int r = work[w];
    const double *c = core + 4 * r;
    StatsAcc &S = st[r];
    if (c[2] != 0.0) {
        S.no_vortex += 1.0;
        S.have_prev = 0;
        return;
    }
    const double a = a_of_rep[r];
    const double x = c[0] * a, y = c[1] * a, rr = sqrt(x * x + y * y);
    S.n += 1.0; S.sx += x; S.sy += y; S.sr2 += x * x + y * y;
    const long long br = (long long)floor(rr / r_max * rb);
    if (br >= 0 && br < rb) hr[(size_t)r * rb + br] += 1ull;
    if (S.have_prev) {
        const double vx = (x - S.px) / dt, vy = (y - S.py) / dt, v = sqrt(vx * vx + vy * vy);
        S.nv += 1.0; S.sv2 += v * v;
        const long long bv = (long long)floor(v / v_max * vb);
        if (bv >= 0 && bv < vb) hv[(size_t)r * vb + bv] += 1ull;
    }
    S.px = x; S.py = y; S.have_prev = 1;
}

cudaError_t launch_stats_update(const int *work, int nwork, const double *core, const double *a_of_rep, StatsAcc *st,
                                unsigned long long *hr, unsigned long long *hv, int rb, int vb, double r_max,
                                double v_max, double dt, cudaStream_t s)
{
    k_stats_update<<<(nwork + 127) / 128, 128, 0, s>>>(work, nwork, core, a_of_rep, st, hr, hv, rb, vb, r_max, v_max, dt);
    return cudaGetLastError();
}

// ----------------------------------------------------------------- <m>

template <typename T>
__global__ void __launch_bounds__(256) k_mean_m(const Replica *reps, const int *work, const T *ybase, double *out)
{
    const int ridx = work[blockIdx.x];
    block_mean<T>(reps[ridx], ybase, out + 3 * ridx);
}

cudaError_t launch_mean_m(int prec, const Replica *reps, const int *work, int nwork, const void *y, double *out,
                          cudaStream_t st)
{
    if (prec == ND_PREC_FP64) k_mean_m<double><<<nwork, 256, 0, st>>>(reps, work, (const double *)y, out);
    else k_mean_m<float><<<nwork, 256, 0, st>>>(reps, work, (const float *)y, out);
    return cudaGetLastError();
}

// -------------------------------------------------------------- schedule

// The time-sliced schedule of a call, written by the GPU in the place of the
// memset of the hand-over words: a call needs no upload and keeps nothing,
// whatever its method and length.  (As tables built by the host and cached per
// class, a change of either cost two allocations, two frees and two blocking
// copies: RK4 and Heun of two steps in turn, 16 x R = 60 nm, 208 -> 167 us a pair,
// 10 x R = 100 nm 298 -> 258; the first Heun call of a new handle 117 -> 93 and
// 149 -> 123.  With the closed form in the stepping kernel itself its registers
// spill: 256 x R = 50 nm, 50 RK4 steps 6.48 -> 6.63 ms.)
__global__ void __launch_bounds__(256) k_schedule(const int *work, int nwork, long long n, int nslots, long long share,
                                                  int room, Segment *segs, int *seg_off, int *flags, int nflags)
{
    const int i = blockIdx.x * 256 + threadIdx.x, slot = i / room, k = i - slot * room;
    for (int f = i; f < nflags; f += gridDim.x * 256) flags[f] = 0;
    if (slot >= nslots) return;
    Segment g;
    const int count = slot_segment(nwork, n, share, slot, k, g);
    if (k < count) {
        g.rep = work[g.pos];
        segs[i] = g;
    }
    if (k == 0) {
        seg_off[2 * slot] = i;
        seg_off[2 * slot + 1] = i + count;
    }
}

cudaError_t launch_schedule(const int *work, int nwork, long long n, int nslots, Segment *segs, int *seg_off, int *flags,
                            int nflags, cudaStream_t st)
{
    const int room = slot_room(nwork, nslots);
    k_schedule<<<(nslots * room + 255) / 256, 256, 0, st>>>(work, nwork, n, nslots, slot_share(nwork, n, nslots), room,
                                                          segs, seg_off, flags, nflags);
    return cudaGetLastError();
}

// ---------------------------------------------------------------- checks

// Sets ND_DEV_NAN in *flag if any component of a cell inside a disk is not
// finite (cells outside the disks and padding columns are ignored).
// grid = (cell blocks, replicas).
template <typename T>
__global__ void k_check_finite(const Replica *reps, const int *work, const T *ybase, unsigned *flag)
{
    const Replica &r = reps[work[blockIdx.y]];
    const int D = r.D, DD = D * D;
    const long long cs = (long long)D * r.Dpad;
    bool bad = false;
    for (int cell = blockIdx.x * blockDim.x + threadIdx.x; cell < DD; cell += gridDim.x * blockDim.x) {
        if (!r.mask[cell]) continue;
        const int j = cell / D, i = cell - j * D;
        const T *y = ybase + r.state_off + (long long)j * r.Dpad + i;
        bad |= !(isfinite(y[0]) && isfinite(y[cs]) && isfinite(y[2 * cs]));
    }
    if (__any_sync(0xffffffffu, bad) && (threadIdx.x & 31) == 0) atomicOr(flag, ND_DEV_NAN);
}

cudaError_t launch_check_finite(int prec, const Replica *reps, const int *work, int nwork, int maxD, const void *y,
                                unsigned *flag, cudaStream_t st)
{
    if (nwork == 0) return cudaSuccess;
    const int cells = maxD * maxD, bx = (cells + 255) / 256 < 64 ? (cells + 255) / 256 : 64;
    dim3 g(bx, nwork);
    if (prec == ND_PREC_FP64) k_check_finite<double><<<g, 256, 0, st>>>(reps, work, (const double *)y, flag);
    else k_check_finite<float><<<g, 256, 0, st>>>(reps, work, (const float *)y, flag);
    return cudaGetLastError();
}

}  // namespace nd
