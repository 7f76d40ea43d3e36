// nd_cluster.cuh -- one replica's time steps, constrained relaxation or field
// on a thread-block cluster of NC CTAs (one per SM): for the sizes P <= 128 when a class has too few replicas
// to fill the GPU with one CTA each, and for P = 192 and 256, whose spectra
// fit in the shared memory of 16 CTAs but not of one.
//
// The replica's rows are split over the cluster: CTA k owns rows
// [k rpc, (k+1) rpc) of the disk (rpc even, so z row pairs stay whole) and
// the column slots [k spc, (k+1) spc) of the P/2 slots of the half spectrum
// (slot 0: the real columns kx = 0 and P/2 packed as one complex column).
// Per field evaluation (Section II.B convolution):
//   1. forward rows: each CTA transforms its own rows (at P = 128 one real
//      row per task at half length, else row pairs) and stores every
//      spectrum entry straight into the shared memory of the CTA that owns
//      its column (st.async into distributed shared memory, counted on the
//      owner's transaction barrier: no thread waits on a remote load or on
//      its own stores);
//   2. each CTA waits until its column slots hold every row;
//   3. columns: one FFT group per (slot, component) transforms its column
//      from local shared memory, applies the spectral kernel (the x and y
//      groups of a column exchange their spectra for the in-plane 2x2 block;
//      the kernel's entries of the CTA's columns are staged in shared memory
//      once per launch), transforms back and stores the rows into the shared
//      memory of their owners (st.async again);
//   4. each CTA waits until its rows hold every column;
//   5. inverse rows and the per-cell epilogue (stage_update) on the CTA's own
//      rows; the next stage's forward rows read only those rows, so a CTA
//      barrier suffices until the next exchange.
// The state y_n, the stage accumulator and the Heun predictor's normals of the
// CTA's rows stay in its shared memory for the whole launch: global memory is
// read once at the start and written once at the end.  The waits on the
// transaction barriers give up after about two seconds, set ND_DEV_TIMEOUT in
// the status word and skip the remaining waits, so a launch always ends.
//
// What bounds it: the chain of one evaluation (rows, exchange, columns,
// exchange, rows, cells), 4.9 us at P = 128 with FP32 and 16 CTAs; in FP64 the
// issue of one warp instruction per 64-76 cycles and sub-partition.  One disk of
// R = 50 nm, 50 Heun steps: 497 us; 16 of R = 60 nm, 50 RK4 steps, time-sliced
// over 15 clusters of 8: 1.24 ms against 4.42 on one CTA each.
#pragma once
#include <cooperative_groups.h>

#include "nd_field_impl.cuh"

namespace nd {

namespace cgc = cooperative_groups;

template <int P, typename T, int NC> struct ClusterGeom {
    static constexpr int G = FFTGeom<P>::G;
    // threads per CTA: enough FFT groups for one per (column slot, component)
    static constexpr int NT = cluster_cta_threads(P);
    static constexpr int NGRP = NT / G;
    static constexpr int SPC = (P / 2) / NC;   // column slots per CTA
    static_assert(SPC >= 1 && (P / 2) % NC == 0, "column slots split evenly over the cluster");
    static_assert(3 * SPC <= NGRP, "one FFT group per (slot, component)");
    static constexpr int KH = SpecGeom<P>::KH;
    // column buffer [3][P/2][SW]: row y of the CTA's SPC column slots, SW = SPC + 1
    // words apart so that a group's column reads fall in different banks, and
    // the lanes of a row group store neighbouring slots of one row
    static constexpr int SW = SPC + 1;
    static constexpr int NTAB = SPC + 1;       // table slots: the CTA's columns, then kx = P/2
};

// Rows per CTA for a grid of D rows: even, so that z row pairs stay in one CTA.
__host__ __device__ __forceinline__ int cluster_rows(int D, int NC) { return 2 * ((D + 2 * NC - 1) / (2 * NC)); }

template <int P, typename T, int NC>
__host__ __device__ __forceinline__ size_t cluster_smem_bytes(int D, int Dpad, bool wbuf)
{
    using CG = ClusterGeom<P, T, NC>;
    const int rpc = cluster_rows(D, NC);
    size_t b = sizeof(cplx<T>) * ((size_t)FFTGeom<P>::R1 * FFTGeom<P>::G               // twiddles
                                  + (size_t)3 * (P / 2) * CG::SW                        // column buffer
                                  + (size_t)3 * rpc * SpecGeom<P>::RS                   // spectrum rows
                                  + (size_t)CG::NGRP * FFTGeom<P>::SCRATCH);            // FFT scratch
    b += sizeof(T) * (size_t)4 * CG::NTAB * CG::KH;                                     // kernel table
    b += sizeof(T) * (size_t)3 * rpc * Dpad * (wbuf ? 4 : 3);   // stage state, y_n, accumulator (+ normals)
    b += 2 * sizeof(int);                                                               // own cell range
    b += 32;                                                                            // mbarriers
    return b;
}

// The spectral step of the packed real columns kx = 0 and P/2 of one
// component after the forward transform of c0 + i c_{P/2}: separation with
// the mirror element, the diagonal kernel entries s0 (kx = 0) and s1
// (kx = P/2) from shared memory, and re-packing for the inverse transform.
// (The entries come halved: they hold the separation's factor 1/2.)
template <int P, typename T>
__device__ __forceinline__ void cluster_packed_scale(cplx<T> *v, const T *s0t, const T *s1t, int t, cplx<T> *scr,
                                                     unsigned gmask)
{
    using Gm = FFTGeom<P>;
    constexpr int G = Gm::G, R1 = Gm::R1;
    mirror_put<P>(v, scr, t);
    __syncwarp(gmask);
#pragma unroll
    for (int o = 0; o < R1; ++o) {
        const int ky = t + G * o;
        const int kyr = ky <= P / 2 ? ky : P - ky;
        const cplx<T> w = mirror_get<P>(scr, ky);
        const cplx<T> F0 = {v[o].x + w.x, v[o].y - w.y};
        const cplx<T> F1 = {v[o].y + w.y, w.x - v[o].x};
        const T s0 = s0t[kyr], s1 = s1t[kyr];
        v[o] = {fm(F0.x, s0, -(F1.y * s1)), fm(F0.y, s0, F1.x * s1)};   // s0 F0 + i s1 F1
    }
    __syncwarp(gmask);
}

// Distributed-shared-memory exchange with transaction barriers: a producer
// stores into another CTA's shared memory with st.async, which also counts
// the bytes on that CTA's mbarrier; the consumer waits until its barrier has
// seen all the bytes it expects.  No producer waits on its own stores, and
// each CTA waits only for the data it reads.
__device__ __forceinline__ uint32_t smem_addr(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ uint32_t cluster_addr(uint32_t a, uint32_t rank)
{
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
    return r;
}
__device__ __forceinline__ void st_async(uint32_t a, cplx<float> v, uint32_t mbar)
{
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v2.f32 [%0], {%1, %2}, [%3];"
                 :: "r"(a), "f"(v.x), "f"(v.y), "r"(mbar) : "memory");
}
__device__ __forceinline__ void st_async(uint32_t a, cplx<double> v, uint32_t mbar)
{
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v2.f64 [%0], {%1, %2}, [%3];"
                 :: "r"(a), "d"(v.x), "d"(v.y), "r"(mbar) : "memory");
}
__device__ __forceinline__ void st_async(uint32_t a, float v, uint32_t mbar)
{
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.f32 [%0], %1, [%2];"
                 :: "r"(a), "f"(v), "r"(mbar) : "memory");
}
__device__ __forceinline__ void st_async(uint32_t a, double v, uint32_t mbar)
{
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.f64 [%0], %1, [%2];"
                 :: "r"(a), "d"(v), "r"(mbar) : "memory");
}
__device__ __forceinline__ void mbar_init(uint32_t mbar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" :: "r"(mbar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect(uint32_t mbar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.release.cta.shared::cta.b64 _, [%0], %1;" :: "r"(mbar), "r"(bytes)
                 : "memory");
}
// Bounded wait for the phase of the given parity to complete, acquiring at
// cluster scope what the producers stored.  Gives up after about two seconds
// of the global timer (a producer that never delivers) and returns false.
__device__ __forceinline__ bool mbar_wait(uint32_t mbar, uint32_t parity)
{
    unsigned long long t0 = 0;
    for (unsigned it = 0; it < (1u << 30); ++it) {
        uint32_t ok;
        asm volatile("{\n\t.reg .pred p;\n\t"
                     "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
                     "selp.u32 %0, 1, 0, p;\n\t}"
                     : "=r"(ok) : "r"(mbar), "r"(parity) : "memory");
        if (ok) return true;
        if ((it & 63) == 63) {
            unsigned long long t;
            asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
            if (t0 == 0) t0 = t;
            else if (t - t0 > 2000000000ull) return false;
        }
    }
    return false;
}

// The constrained relaxation (MODE == M_RELAX): the sweep of k_fused.  Its
// schedule is a queue of turns: ticket k takes turn k / nwork of replica
// work[k % nwork] -- at most `quantum` sweeps -- once the replica's turn
// before that is over (flags[rep] counts them; that turn's ticket is lower, so
// its cluster is running).  Converged replicas are passed over, and the
// clusters leave when all have converged or used up their sweeps.  With no
// more replicas than clusters a turn is the whole relaxation.
//
// The torque m x e is what the sweep drives to zero, so it is evaluated from
// small terms: the exchange as sum_j (m_j - m_i) over the neighbours inside
// the disk, straight from the state (the edge rows of the neighbouring CTAs
// arrive as halos), and the demagnetisation alone through the FFT.  With the
// exchange folded into the FFT, whose rounding is relative to |b| ~ 4, the
// residual of an FP32 sweep carried noise of ~5e-7 and replicas stopped up to
// ten sweeps from where FP64 arithmetic stops.
//
// Above P = 128 in FP32 (WIDE) more replicas relax in grid-wide passes, which add
// their CTAs' sums, take the Newton step and hold the multipliers in FP64.  Here
// the warps' sums are added in pairs, at most ten FP32 additions deep (there
// twelve), and the rest is computed and held in pairs of floats (Two, some 46
// bits): FP64 issues a warp instruction in 64-76 cycles, and this is a chain that
// every CTA waits for.  All of it in FP64 cost 0.5-0.8 us of a sweep of 13.8
// (R = 100 nm), this 0.3 (0.15 of 11.8 at 70 nm, 0.2 of 14.5 at 128 nm).
// Multipliers of R = 70, 100 and 128 nm after 400 sweeps, against FP64: 2.7e-8,
// 3.5e-8 and 2.9e-8 off, as with FP64 in this place; grid-wide 1.4e-7, 2.3e-7,
// 1.6e-7; with FP32 in this place 1.2e-7, 4.8e-8, 3.2e-8.
struct ClusterRelax {
    RelaxIO *rio;
    const double *twP64;   // exp(-2 pi i k / P), FP64
    double eta, tol, rc2;
    int max_iter, quantum, nwork;
    int *ndone;   // replicas finished
};

// Without SEG, one replica per cluster for the whole launch (compiled apart:
// the schedule's loop around the steps cost 5-10% of each step).  With SEG
// (more replicas than clusters fit on the GPU), a time-sliced schedule: the cluster
// with ticket i (tickets count the clusters in the order they start, so every
// cluster that another one waits for is already running) runs the segments
// segs[seg_off[2i] .. seg_off[2i+1]), passing replicas on through flags.
template <int P, typename T, int MODE, int NC, bool SEG>
__global__ void __launch_bounds__(ClusterGeom<P, T, NC>::NT, 1)
    k_cluster(const Replica *__restrict__ reps, const int *__restrict__ work, T *__restrict__ ybase, T *__restrict__ outbase,
              const cplx<T> *__restrict__ twP, long long nsteps_all, unsigned long long step_base, int use_wbuf,
              unsigned *__restrict__ status, const Segment *__restrict__ segs, const int *__restrict__ seg_off,
              int *__restrict__ flags, int *__restrict__ ticket, int wait_polls, const ClusterRelax rx)
{
    using Gm = FFTGeom<P>;
    using CG = ClusterGeom<P, T, NC>;
    constexpr int G = Gm::G, R1 = Gm::R1, RS = SpecGeom<P>::RS, KH = CG::KH, NT = CG::NT, NGRP = CG::NGRP;
    constexpr int SPC = CG::SPC, SW = CG::SW, NTAB = CG::NTAB;
    static_assert(MODE == M_RELAX ? SEG : (MODE == M_FIELD ? !SEG : true), "turns or one launch per replica");
    constexpr bool RELAX = MODE == M_RELAX, WIDE = RELAX && sizeof(T) == 4 && P > 128;
    cgc::cluster_group cluster = cgc::this_cluster();
    const int rank = (int)cluster.block_rank();
    extern __shared__ __align__(16) unsigned char smem[];
    const int tid = threadIdx.x;
    GroupId<P> gid(tid);
    unsigned long long *mbars = reinterpret_cast<unsigned long long *>(smem);   // [0] columns, [1] rows, [2] [3] sums
    const uint32_t mb_col = smem_addr(mbars), mb_row = smem_addr(mbars + 1), mb_sum = smem_addr(mbars + 2);
    __shared__ unsigned long long halo_bar;
    const uint32_t mb_halo = smem_addr(&halo_bar);
    cplx<T> *tw = reinterpret_cast<cplx<T> *>(smem + 32);
    __shared__ RelaxAcc<T> racc[RELAX ? NT / 32 : 1];   // per warp
    // Per CTA of the cluster, for even and odd sweeps: a CTA without rows waits
    // for no field of the others, so its sums of the next sweep may reach another
    // such CTA before a third one's of this sweep.  It cannot be two sweeps ahead
    // (it needs everyone's sums to go on).
    __shared__ T rpart[2][RELAX ? NC : 1][6];
    __shared__ T lam_s[2];
    __shared__ int conv_s;
    __shared__ int bcast;   // rank 0's: the cluster's ticket, then whether a hand-over arrived
    load_twiddles<P>(tw, twP, tid, NT);
    if (tid == 0) {
        mbar_init(mb_col, 1);
        mbar_init(mb_row, 1);
        mbar_init(mb_sum, 1);
        mbar_init(mb_sum + 8, 1);
        if (RELAX) mbar_init(mb_halo, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        if (SEG && !RELAX && rank == 0) bcast = atomicAdd(ticket, 1);
    }
    cluster.sync();   // every CTA runs, with its barriers initialised, before the first remote store
    const int slot = SEG && !RELAX ? *cluster.map_shared_rank(&bcast, 0) : 0;
    uint32_t phase = 0, hphase = 0, sweep = 0;   // sweep: of the launch, over all its turns
    bool bailed = false;   // this thread's wait ran out once: it skips every later wait
    // Only launches that share the counter (calls of one handle that overlap) draw
    // a ticket beyond the schedule: such a cluster has nothing to run.
    const bool beyond = SEG && !RELAX && slot >= (int)(gridDim.x / NC);
    if (beyond && rank == 0 && tid == 0) atomicOr(status, ND_DEV_ORDER);
    const int sg_begin = SEG && !RELAX && !beyond ? seg_off[2 * slot] : 0;
    const int sg_end = RELAX ? 0x7fffffff : beyond ? 0 : SEG ? seg_off[2 * slot + 1] : 1;
    for (int sg = sg_begin; sg < sg_end; ++sg) {
    Segment seg;
    if constexpr (RELAX) {
        // rank 0 takes the next turn of a replica that has not finished: -1 none left, -2 a wait expired
        cluster.sync();
        if (rank == 0 && tid == 0) {
            int got = -1;
            while (atomicAdd(rx.ndone, 0) < rx.nwork) {
                const int k = atomicAdd(ticket, 1), rep = work[k % rx.nwork], turn = k / rx.nwork;
                if ((long long)turn * rx.quantum >= rx.max_iter) break;
                bool ok = false;
                for (int it = 0; it < wait_polls && !ok; ++it) {
                    ok = atomicAdd(flags + rep, 0) >= turn;
                    if (!ok) __nanosleep(256);
                }
                if (!ok) {
                    atomicOr(status, ND_DEV_TIMEOUT);
                    got = -2;
                    break;
                }
                __threadfence();
                if (__ldcg(&rx.rio[rep].status) != 0) {
                    got = rep;
                    break;
                }
                atomicExch(flags + rep, 0x7fffffff);   // finished: its later turns wait for nothing
            }
            bcast = got;
        }
        cluster.sync();
        seg = Segment{*cluster.map_shared_rank(&bcast, 0), 0, 1, 0, 0, 0};
        if (seg.rep < 0) break;   // (the same for every CTA of the cluster)
        seg.nsteps = min(rx.quantum, rx.max_iter - __ldcg(&rx.rio[seg.rep].iters));
    } else if constexpr (SEG) {
        seg = segs[sg];
    } else {
        seg = Segment{work[blockIdx.x / NC], 0, 0, 0, 0, nsteps_all};
    }
    const long long nsteps = seg.nsteps;
    const Replica &r = reps[seg.rep];
    if (SEG && !RELAX) {   // (the same for every CTA of the cluster)
        cluster.sync();   // the ticket is read; the previous segment's rows and columns are no longer used
        if (rank == 0 && tid == 0) {
            bcast = seg.wait ? (int)wait_flag(flags + seg.rep, wait_polls) : 1;
            if (!bcast) atomicOr(status, ND_DEV_TIMEOUT);
        }
        cluster.sync();
        if (!*cluster.map_shared_rank(&bcast, 0)) break;
    }
    const int D = r.D, Dpad = r.Dpad, rpc = cluster_rows(D, NC);
    const int ylo = rank * rpc, nloc = max(0, min(D, ylo + rpc) - ylo);   // this CTA's rows [ylo, ylo + nloc)
    const long long lcs = (long long)rpc * RS;                            // local spectrum component stride
    const long long lms = (long long)rpc * Dpad;                          // local state component stride
    const long long ms_s = (long long)D * Dpad;                           // global state component stride
    cplx<T> *colbuf = tw + R1 * G;                                        // [3][P/2][SW]
    cplx<T> *spec = colbuf + 3 * (P / 2) * SW;                            // [3][rpc][RS]
    cplx<T> *scratch = spec + 3 * lcs;
    T *gtab = reinterpret_cast<T *>(scratch + NGRP * Gm::SCRATCH);        // [4][NTAB][KH]
    T *msl = gtab + 4 * NTAB * KH;                                        // [3][rpc][Dpad]
    T *ynl = msl + 3 * lms, *accl = ynl + 3 * lms;
    T *wl = use_wbuf ? accl + 3 * lms : nullptr;
    int *crange = reinterpret_cast<int *>((use_wbuf ? wl : accl) + 3 * lms);
    cplx<T> *scr = scratch + gid.group * Gm::SCRATCH;
    const V3Ptr<T> ms{msl, lms}, wb{wl, lms}, ynv{ynl, lms}, accv{accl, lms}, none{nullptr, 0};
    const V3Ptr<T> yg{ybase + r.state_off, ms_s};
    // the state of the CTA's rows (zero outside the disk)
    for (int i = tid; i < nloc * D; i += NT) {
        const int lr = i / D, x = i - lr * D, y = ylo + lr;
        const long long si = (long long)y * Dpad + x, mi = (long long)lr * Dpad + x;
        const vec3<T> m0 = r.mask[y * D + x] ? yg.ldcg(si) : vec3<T>{T(0), T(0), T(0)};
        ms.st(mi, m0);
        ynv.st(mi, m0);
    }
    // the kernel's entries of the CTA's columns (and of kx = P/2), from the
    // component-major copy of the table
    {
        constexpr int KK = KH * KH;
        const T *Gc = reinterpret_cast<const T *>(r.Ghat) + 4 * KK;
        for (int i = tid; i < 4 * NTAB * KH; i += NT) {
            const int c = i / (NTAB * KH), rem = i - c * (NTAB * KH), j = rem / KH, ky = rem - j * KH;
            const int kx = j < SPC ? rank * SPC + j : P / 2;
            // with the factors 1/2 of the separations of row pairs and of the
            // packed columns: powers of two, so the rounding is that of the
            // other kernels, which apply them where they separate
            const T half = (HalfRows<P>::on ? T(1) : T(0.5)) * (kx == 0 || kx == P / 2 ? T(0.5) : T(1));
            if constexpr (RELAX) {   // without the exchange
                const double g = __ldg(r.Ghat64 + (long long)(4 + c) * KK + kx * KH + ky);
                const double ex = c == 2 ? 0.0 : 2.0 * (__ldg(rx.twP64 + 2 * kx) + __ldg(rx.twP64 + 2 * ky));
                gtab[i] = half * (T)fm(-ex, 1.0 / ((double)P * P), g);
            } else {
                gtab[i] = half * __ldg(Gc + (long long)c * KK + kx * KH + ky);
            }
        }
    }
    // relaxation: the rows of the neighbouring CTAs above and below, zero where there are none
    T *const halo = wl;   // [2][3][Dpad]
    const bool up = RELAX && rank > 0 && nloc > 0, down = RELAX && nloc > 0 && ylo + nloc < D;
    if constexpr (RELAX) {
        for (int i = tid; i < 2 * Dpad; i += NT) {
            const int h = i / Dpad, x = i - h * Dpad, y = h ? ylo + nloc : ylo - 1;
            const bool in = (h ? down : up) && x < D && r.mask[y * D + x];
            V3Ptr<T>{halo + h * 3 * Dpad, Dpad}.st(x, in ? yg.ldcg((long long)y * Dpad + x) : vec3<T>{T(0), T(0), T(0)});
        }
    }
    // the CTA's cells: a contiguous range of the ascending cell list
    if (tid == 0) {
        int lo = 0, hi = r.ncells;
        while (lo < hi) { const int mid = (lo + hi) >> 1; if (__ldg(r.cells + mid) < ylo * D) lo = mid + 1; else hi = mid; }
        crange[0] = lo;
        hi = r.ncells;
        while (lo < hi) { const int mid = (lo + hi) >> 1; if (__ldg(r.cells + mid) < (ylo + nloc) * D) lo = mid + 1; else hi = mid; }
        crange[1] = lo;
    }
    // row tasks of this CTA: one real row per (component, row) at P = 128
    // (half-length transforms), else xy rows 0..nloc-1, then z pairs (0,1), ...
    constexpr bool HR = HalfRows<P>::on;
    const int nrt = HR ? 3 * nloc : nloc + (nloc + 1) / 2;
    const int nrounds = (nrt + NGRP - 1) / NGRP;
    // column task of this group: slot j (column kx = rank SPC + j, slot 0 of
    // rank 0 being the packed pair), component c
    const int cj = gid.group % SPC, cc = gid.group / SPC;
    const bool ctask = gid.group < 3 * SPC;   // groups beyond 3 SPC idle in the column pass
    const int kslot = rank * SPC + cj;
    const bool packed = ctask && kslot == 0;
    // bytes each CTA receives from the other CTAs per stage (what it sends to
    // itself goes by plain stores, made visible by a CTA barrier): its SPC
    // column slots of every other CTA's rows, and the P/2 + 1 spectrum entries
    // of each own row from the other CTAs' column slots (rank 0 holds the
    // packed pair: SPC + 1 entries of its own)
    const uint32_t bytes_col = (uint32_t)(3 * (D - nloc) * SPC * sizeof(cplx<T>));
    const uint32_t bytes_row = (uint32_t)(3 * nloc * (P / 2 + 1 - SPC - (rank == 0 ? 1 : 0)) * sizeof(cplx<T>));
    T relX = T(0), relY = T(0);
    Two lam2 = {0.0f, 0.0f};   // WIDE: multiplier tid of threads 0 and 1
    if constexpr (RELAX) {
        const RelaxIO *io = rx.rio + seg.rep;
        relX = (T)io->X[0];
        relY = (T)io->X[1];
        if (tid == 0) {
            lam_s[0] = (T)__ldcg(&io->lam[0]);
            lam_s[1] = (T)__ldcg(&io->lam[1]);
            conv_s = 0;
        }
        if (WIDE && tid < 2) {
            const double l = __ldcg(&io->lam[tid]);
            lam2.hi = (float)l;
            lam2.lo = (float)(l - (double)lam2.hi);
        }
    }
    __syncthreads();   // the state, the kernel's entries and the cell range are in place
    const int c0 = crange[0], c1 = crange[1];
    T *const zl = reinterpret_cast<T *>(scratch);   // relaxation: neighbour counts (the FFT scratch is idle then)
    T res_last = T(0);   // thread 0: the last sweep's residual
    long long n = 0;

    for (n = 0; n < nsteps; ++n) {
        const unsigned long long step = step_base + r.step0 + (unsigned long long)(seg.step_begin + n);
        for (int stage = 0; stage < ModeStages<MODE>::n; ++stage) {
            if (tid == 0) {
                mbar_expect(mb_col, bytes_col);
                mbar_expect(mb_row, bytes_row);
                if (RELAX) mbar_expect(mb_sum + 8 * (sweep & 1), (uint32_t)((NC - 1) * 6 * sizeof(T)));
            }
            // 1. forward rows of the CTA's own rows, sent to the column owners
            if constexpr (HR) {
                for (int q = gid.group; q < nrounds * NGRP; q += NGRP) {
                    const bool act = q < nrt;
                    const int c = act ? q / nloc : 0, l = act ? q - c * nloc : 0, y = ylo + l;
                    cplx<T> v[FFTGeom<P / 2>::R1];
                    T xm;
                    row_fwd_half_spectrum<P, T>(act, msl + c * lms + (long long)l * Dpad, D, v, xm, gid.t, scr, tw,
                                                gid.gmask);
                    if (act) {
#pragma unroll
                        for (int o = 0; o < FFTGeom<P / 2>::R1; ++o) {
                            const int k = gid.t + G * o;   // k = 0 goes with k = P/2 into the packed slot
                            const int ow = k / SPC, j = k - ow * SPC;
                            const cplx<T> a = k == 0 ? cplx<T>{v[o].x, xm} : v[o];
                            const int i = (c * (P / 2) + y) * SW + j;
                            if (ow == rank) {
                                colbuf[i] = a;
                            } else {
                                st_async(cluster_addr(smem_addr(colbuf), ow) + (uint32_t)(i * sizeof(cplx<T>)), a,
                                         cluster_addr(mb_col, ow));
                            }
                        }
                    }
                }
            } else
            for (int q = gid.group; q < nrounds * NGRP; q += NGRP) {
                const bool act = q < nrt;
                const bool isxy = q < nloc;
                const int l0 = isxy ? q : 2 * (q - nloc), l1 = l0 + 1;
                const bool hasB = isxy || (l1 < nloc);
                cplx<T> v[R1];
#pragma unroll
                for (int o = 0; o < R1; ++o) v[o] = {T(0), T(0)};
#pragma unroll
                for (int o = 0; o < R1 / 2; ++o) {
                    const int x = gid.t + G * o;
                    if (act && x < D) {
                        if (isxy) v[o] = {msl[(long long)l0 * Dpad + x], msl[lms + (long long)l0 * Dpad + x]};
                        else v[o] = {msl[2 * lms + (long long)l0 * Dpad + x],
                                     hasB ? msl[2 * lms + (long long)l1 * Dpad + x] : T(0)};
                    }
                }
                fft_group<P, -1, FFT_HALF_IN>(v, gid.t, scr, tw, gid.gmask);
                mirror_put<P>(v, scr, gid.t);
                __syncwarp(gid.gmask);
                if (act) {
                    // A: the row ending in the real part (x, or the first z row),
                    // B: the one ending in the imaginary part (y, or the second z row)
                    const int cA = isxy ? 0 : 2, cB = isxy ? 1 : 2;
                    const int yA = ylo + l0, yB = isxy ? ylo + l0 : ylo + l1;
                    T rA0 = T(0), rB0 = T(0);   // lane t = 0: the real entries at k = 0 (then k = P/2)
#pragma unroll
                    for (int o = 0; o < R1; ++o) {
                        const int k = gid.t + G * o;
                        if (k <= P / 2) {
                            const cplx<T> w = mirror_get<P>(scr, k);
                            // twice the spectra (the kernel's entries are halved)
                            const cplx<T> A = {v[o].x + w.x, v[o].y - w.y};
                            const cplx<T> B = {v[o].y + w.y, w.x - v[o].x};
                            if (k == 0) {
                                rA0 = A.x;
                                rB0 = B.x;
                            } else {
                                const int ow = k == P / 2 ? 0 : k / SPC, j = k == P / 2 ? 0 : k - ow * SPC;
                                const cplx<T> a = k == P / 2 ? cplx<T>{rA0, A.x} : A;
                                const cplx<T> b2 = k == P / 2 ? cplx<T>{rB0, B.x} : B;
                                const int iA = (cA * (P / 2) + yA) * SW + j, iB = (cB * (P / 2) + yB) * SW + j;
                                if (ow == rank) {
                                    colbuf[iA] = a;
                                    if (hasB) colbuf[iB] = b2;
                                } else {
                                    const uint32_t base = cluster_addr(smem_addr(colbuf), ow);
                                    const uint32_t mb = cluster_addr(mb_col, ow);
                                    st_async(base + (uint32_t)(iA * sizeof(cplx<T>)), a, mb);
                                    if (hasB) st_async(base + (uint32_t)(iB * sizeof(cplx<T>)), b2, mb);
                                }
                            }
                        }
                    }
                }
                __syncwarp(gid.gmask);
            }
            // every row spectrum of this CTA's columns has arrived (the
            // barrier makes the CTA's own plain stores visible)
            if (!bailed && !mbar_wait(mb_col, phase & 1)) {
                bailed = true;
                atomicOr(status, ND_DEV_TIMEOUT);
            }
            __syncthreads();
            // 3. columns from the local column buffer, back to the row owners
            {
                cplx<T> v[R1];
#pragma unroll
                for (int o = 0; o < R1; ++o) v[o] = {T(0), T(0)};
                const int kx = packed ? 0 : kslot;
                if (ctask) {
                    const cplx<T> *col = colbuf + cc * (P / 2) * SW + cj;
#pragma unroll
                    for (int o = 0; o < R1 / 2; ++o) {
                        const int y = gid.t + G * o;
                        if (y < D) v[o] = col[y * SW];
                    }
                }
                // one transform call for both kinds of column, so that a warp
                // holding the packed slot does not run two transforms in turn
                if (ctask) fft_group<P, -1, FFT_HALF_IN>(v, gid.t, scr, tw, gid.gmask);
                if (packed) {
                    const int comp = cc == 2 ? 3 : cc;   // the diagonal entry: xx, yy or zz
                    cluster_packed_scale<P, T>(v, gtab + (comp * NTAB) * KH, gtab + (comp * NTAB + SPC) * KH, gid.t,
                                               scr, gid.gmask);
                }
                // the x and y groups of a column exchange their spectra
                if (ctask && !packed && cc < 2) {
#pragma unroll
                    for (int o = 0; o < R1; ++o) scr[o * G + gid.t] = v[o];
                }
                __syncthreads();
                if (ctask && !packed) {
                    if (cc < 2) {
                        const cplx<T> *other = scratch + ((1 - cc) * SPC + cj) * Gm::SCRATCH;
                        const T *gd = gtab + (cc * NTAB + cj) * KH, *go = gtab + (2 * NTAB + cj) * KH;
#pragma unroll
                        for (int o = 0; o < R1; ++o) {
                            const int ky = gid.t + G * o;
                            const bool up = ky <= P / 2;
                            const int kyr = up ? ky : P - ky;
                            const T gdiag = gd[kyr], gxy0 = go[kyr];
                            const T gxy = up ? gxy0 : -gxy0;   // G_xy is odd in ky
                            const cplx<T> w = other[o * G + gid.t];
                            v[o] = cc == 0 ? tensor_row(gdiag, v[o], gxy, w) : tensor_row(gxy, w, gdiag, v[o]);
                        }
                    } else {
                        const T *gz = gtab + (3 * NTAB + cj) * KH;
#pragma unroll
                        for (int o = 0; o < R1; ++o) {
                            const int ky = gid.t + G * o;
                            const int kyr = ky <= P / 2 ? ky : P - ky;
                            v[o] = cscale(v[o], gz[kyr]);
                        }
                    }
                }
                __syncthreads();   // the partners' spectra are read before the scratch is reused
                if (ctask) fft_group<P, +1, FFT_HALF_OUT>(v, gid.t, scr, tw, gid.gmask);
#pragma unroll
                for (int o = 0; o < R1 / 2; ++o) {
                    const int y = gid.t + G * o;
                    if (ctask && y < D) {
                        const int ow = y / rpc, lr = y - ow * rpc;   // the row's owner
                        cplx<T> *dst = spec + cc * lcs + (long long)lr * RS;
                        if (ow == rank) {
                            if (packed) {
                                dst[0] = {v[o].x, T(0)};
                                dst[P / 2] = {v[o].y, T(0)};
                            } else {
                                dst[kx] = v[o];
                            }
                        } else {
                            const uint32_t row = cluster_addr(smem_addr(dst), ow);
                            const uint32_t mb = cluster_addr(mb_row, ow);
                            if (packed) {
                                st_async(row, cplx<T>{v[o].x, T(0)}, mb);
                                st_async(row + (uint32_t)((P / 2) * sizeof(cplx<T>)), cplx<T>{v[o].y, T(0)}, mb);
                            } else {
                                st_async(row + (uint32_t)(kx * sizeof(cplx<T>)), v[o], mb);
                            }
                        }
                    }
                }
            }
            // every column entry of this CTA's rows has arrived
            if (!bailed && !mbar_wait(mb_row, phase & 1)) {
                bailed = true;
                atomicOr(status, ND_DEV_TIMEOUT);
            }
            __syncthreads();
            ++phase;
            // 5. inverse rows of the CTA's own rows (the field rows, in place)
            if constexpr (HR) {
                for (int q = gid.group; q < nrounds * NGRP; q += NGRP) {
                    const bool act = q < nrt;
                    const int c = act ? q / nloc : 0, l = act ? q - c * nloc : 0;
                    cplx<T> *row = spec + c * lcs + (long long)l * RS;
                    row_inv_half<P, T>(act, row, D, reinterpret_cast<T *>(row), gid.t, scr, tw, gid.gmask);
                }
            } else
            for (int q = gid.group; q < nrounds * NGRP; q += NGRP) {
                const bool act = q < nrt;
                const bool isxy = q < nloc;
                const int l0 = isxy ? q : 2 * (q - nloc), l1 = l0 + 1;
                const bool hasB = isxy || (l1 < nloc);
                cplx<T> *rA = isxy ? spec + (long long)l0 * RS : spec + 2 * lcs + (long long)l0 * RS;
                cplx<T> *rB = isxy ? spec + lcs + (long long)l0 * RS : spec + 2 * lcs + (long long)l1 * RS;
                cplx<T> v[R1];
                row_inv_fft<P, T>(v, act, rA, rB, hasB, gid.t, scr, tw, gid.gmask);
                if (act) {
                    T *oA = reinterpret_cast<T *>(rA), *oB = reinterpret_cast<T *>(rB);
#pragma unroll
                    for (int o = 0; o < R1 / 2; ++o) {
                        const int x = gid.t + G * o;
                        if (x < D) {
                            oA[x] = v[o].x;
                            if (hasB) oB[x] = v[o].y;
                        }
                    }
                }
            }
            __syncthreads();
            if constexpr (RELAX) {
                // the sweep of k_fused's relaxation mode: trial alignment with the
                // current multipliers (kept in the accumulator for the cells that
                // they do not touch), sums over the cluster, one Newton step by
                // every CTA alike, then the update
                const StepParams<T> sp = step_params<T>(r);
                const T *hr = reinterpret_cast<const T *>(spec);
                const T eta = (T)rx.eta, rc2 = (T)rx.rc2, half = T(0.5) * (T)(D - 1);
                const T l0 = lam_s[0], l1 = lam_s[1];
                if (n > 0) {   // (the first sweep's halos were read from the caller's state)
                    if (!bailed && !mbar_wait(mb_halo, hphase & 1)) {
                        bailed = true;
                        atomicOr(status, ND_DEV_TIMEOUT);
                    }
                    ++hphase;
                }
                RelaxAcc<T> a = {T(0), T(0), T(0), T(0), T(0), T(0)};
                const vec3<T> zero3 = {T(0), T(0), T(0)};
                for (int k = c0 + tid; k < c1; k += NT) {
                    const int cell = __ldg(r.cells + k), y = cell / D, x = cell - y * D, lr = y - ylo;
                    const long long mi = (long long)lr * Dpad + x, hi = (long long)lr * (2 * RS) + x;
                    const vec3<T> m = ms.ld(mi);
                    vec3<T> e = {hr[hi] + sp.chext[0], hr[2 * lcs + hi] + sp.chext[1], hr[4 * lcs + hi] + sp.chext[2]};
                    T z = T(0);   // neighbours inside the disk (cells outside hold zero)
                    auto add = [&](vec3<T> q) {
                        const bool in = q.x != T(0) || q.y != T(0) || q.z != T(0);
                        z += in ? T(1) : T(0);
                        e.x += in ? q.x - m.x : T(0);
                        e.y += in ? q.y - m.y : T(0);
                        e.z += in ? q.z - m.z : T(0);
                    };
                    add(x > 0 ? ms.ld(mi - 1) : zero3);
                    add(x + 1 < D ? ms.ld(mi + 1) : zero3);
                    add(lr > 0 ? ms.ld(mi - Dpad) : V3Ptr<T>{halo, Dpad}.ld(x));
                    add(lr + 1 < nloc ? ms.ld(mi + Dpad) : V3Ptr<T>{halo + 3 * Dpad, Dpad}.ld(x));
                    const T dx = (T)x - half - relX, dy = (T)y - half - relY;
                    // (y_n's place keeps e for the second alignment, the normals' the halos)
                    ynv.st(mi, e);
                    accv.st(mi, relax_cell<T>(m, e, fm(dx, dx, dy * dy) < rc2, dx, dy, l0, l1, eta, a, z));
                    zl[mi] = z;
                }
                a.C0 = warp_sum_t(a.C0); a.C1 = warp_sum_t(a.C1); a.J00 = warp_sum_t(a.J00);
                a.J01 = warp_sum_t(a.J01); a.J11 = warp_sum_t(a.J11); a.res = warp_max_t(a.res);
                if ((tid & 31) == 0) racc[tid >> 5] = a;
                __syncthreads();
                T(*const rp)[6] = rpart[sweep & 1];
                const uint32_t mb_red = mb_sum + 8 * (sweep & 1);
                if (tid < 6 * NC) {   // value v of this CTA to CTA q
                    const int q = tid / 6, v = tid - 6 * q;
                    T t = (&racc[0].C0)[v];
                    if constexpr (WIDE) {
                        T u[NT / 32];
#pragma unroll
                        for (int w = 0; w < NT / 32; ++w) u[w] = (&racc[w].C0)[v];
#pragma unroll
                        for (int o = 1; o < NT / 32; o *= 2)
#pragma unroll
                            for (int w = 0; w < NT / 32; w += 2 * o) u[w] = v == 5 ? max(u[w], u[w + o]) : u[w] + u[w + o];
                        t = u[0];
                    } else {
                        for (int w = 1; w < NT / 32; ++w) {
                            const T u = (&racc[w].C0)[v];
                            t = v == 5 ? max(t, u) : t + u;
                        }
                    }
                    if (q == rank) rp[q][v] = t;
                    else st_async(cluster_addr(smem_addr(&rp[rank][v]), q), t, cluster_addr(mb_red, q));
                }
                __syncthreads();
                if (tid < 32) {
                    if (!bailed && !mbar_wait(mb_red, (sweep >> 1) & 1)) {
                        bailed = true;
                        atomicOr(status, ND_DEV_TIMEOUT);
                    }
                    if constexpr (WIDE) {
                        // lanes 4v..4v+3 add value v's partial sums
                        const int v = min(tid >> 2, 5), q0 = tid & 3;
                        Two t = {rp[q0][v], 0.0f};
                        T res = rp[q0][5];
#pragma unroll
                        for (int q = q0 + 4; q < q0 + NC; q += 4) {
                            t.lo += two_sum(t.hi, rp[q][v]);
                            res = max(res, rp[q][5]);
                        }
#pragma unroll
                        for (int o = 1; o < 4; o *= 2) {
                            const float h = __shfl_xor_sync(0xffffffffu, t.hi, o), l = __shfl_xor_sync(0xffffffffu, t.lo, o);
                            t.lo += l + two_sum(t.hi, h);
                            res = max(res, __shfl_xor_sync(0xffffffffu, res, o));
                        }
                        auto sum = [&](int k) {
                            return Two{__shfl_sync(0xffffffffu, t.hi, 4 * k), __shfl_sync(0xffffffffu, t.lo, 4 * k)};
                        };
                        const Two C0 = sum(0), C1 = sum(1), J00 = sum(2), J01 = sum(3), J11 = sum(4);
                        // lanes 0 and 1 a numerator each, lane 2 the determinant
                        const Two n = two_det(tid == 0 ? J11 : J00, tid == 0 ? C0 : tid == 1 ? C1 : J11, J01,
                                              tid == 0 ? C1 : tid == 1 ? C0 : J01);
                        const float dh = __shfl_sync(0xffffffffu, n.hi, 2), dl = __shfl_sync(0xffffffffu, n.lo, 2);
                        if (tid < 2) {   // a multiplier each
                            res_last = res;
                            if (res < (T)rx.tol) {
                                conv_s = 1;
                            } else {
                                const float rd = 1.0f / dh, q = n.hi * rd;
                                const float q2 = (fm(-q, dh, n.hi) + fm(-q, dl, n.lo)) * rd;
                                if (dh != 0.0f && isfinite(dh)) {   // lam -= q + q2
                                    lam2.lo += two_sum(lam2.hi, -q) - q2;
                                    lam2.lo = two_sum(lam2.hi, lam2.lo);
                                }
                                lam_s[tid] = lam2.hi;
                            }
                        }
                    } else {
                    const int v = min(tid, 5);
                    T t = rp[0][v];
                    for (int q = 1; q < NC; ++q) t = v == 5 ? max(t, rp[q][v]) : t + rp[q][v];
                    const T C0 = __shfl_sync(0xffffffffu, t, 0), C1 = __shfl_sync(0xffffffffu, t, 1);
                    const T J00 = __shfl_sync(0xffffffffu, t, 2), J01 = __shfl_sync(0xffffffffu, t, 3);
                    const T J11 = __shfl_sync(0xffffffffu, t, 4), res = __shfl_sync(0xffffffffu, t, 5);
                    if (tid == 0) {
                        res_last = res;
                        if (res < (T)rx.tol) {
                            conv_s = 1;
                        } else {
                            const T det = fm(J00, J11, -(J01 * J01));
                            if (det != T(0) && isfinite(det)) {
                                lam_s[0] += -fm(J11, C0, -(J01 * C1)) / det;
                                lam_s[1] += -fm(J00, C1, -(J01 * C0)) / det;
                            }
                        }
                    }
                    }
                }
                __syncthreads();
                ++sweep;
                if (conv_s) break;   // leaves the stage loop; the sweep loop stops below
                const T m0 = lam_s[0], m1 = lam_s[1];
                for (int k = c0 + tid; k < c1; k += NT) {
                    const int cell = __ldg(r.cells + k), y = cell / D, x = cell - y * D, lr = y - ylo;
                    const long long mi = (long long)lr * Dpad + x;
                    const T dx = (T)x - half - relX, dy = (T)y - half - relY;
                    vec3<T> mp = accv.ld(mi);   // this thread's own store
                    if (fm(dx, dx, dy * dy) < rc2) {
                        RelaxAcc<T> dummy = {T(0), T(0), T(0), T(0), T(0), T(0)};
                        mp = relax_cell<T>(ms.ld(mi), ynv.ld(mi), true, dx, dy, m0, m1, eta, dummy, zl[mi]);
                    }
                    ms.st(mi, mp);
                }
                __syncthreads();
                if (n + 1 < nsteps) {   // the edge rows to the neighbours (which have read theirs: their sums arrived)
                    if (tid == 0) mbar_expect(mb_halo, (uint32_t)((int)up + (int)down) * 3 * D * sizeof(T));
                    for (int i = tid; i < 3 * D; i += NT) {
                        const int c = i / D, x = i - c * D;
                        if (up)   // my first row is the row below the CTA above
                            st_async(cluster_addr(smem_addr(halo + (3 + c) * Dpad + x), rank - 1),
                                     msl[c * lms + x], cluster_addr(mb_halo, rank - 1));
                        if (down)
                            st_async(cluster_addr(smem_addr(halo + c * Dpad + x), rank + 1),
                                     msl[c * lms + (long long)(nloc - 1) * Dpad + x], cluster_addr(mb_halo, rank + 1));
                    }
                }
                continue;
            }
            const StepParams<T> sp = step_params<T>(r);
            const T *hr = reinterpret_cast<const T *>(spec);
            if constexpr (MODE == M_FIELD) {   // the CTA's rows of the output, zero outside the disk
                const V3Ptr<T> out{outbase + r.state_off + (long long)ylo * Dpad, ms_s};
                for (int i = tid; i < nloc * Dpad; i += NT) {
                    const int lr = i / Dpad, x = i - lr * Dpad, hi = lr * (2 * RS) + x;
                    const bool in = x < D && r.mask[(ylo + lr) * D + x];
                    out.st(i, in ? vec3<T>{hr[hi] + sp.chext[0], hr[2 * lcs + hi] + sp.chext[1], hr[4 * lcs + hi] + sp.chext[2]}
                                 : vec3<T>{T(0), T(0), T(0)});
                }
                continue;
            }
            // the per-cell epilogue of the CTA's cells
            const vec3<T> cx = step_chext<T>(r, sp, step);
            if constexpr (!RELAX && MODE != M_FIELD)
            for (int k = c0 + tid; k < c1; k += NT) {
                const int cell = __ldg(r.cells + k);
                const int y = cell / D, x = cell - y * D, lr = y - ylo;
                const long long mi = (long long)lr * Dpad + x;
                const long long hi = (long long)lr * (2 * RS) + x;
                const vec3<T> b = {hr[hi] + cx.x, hr[2 * lcs + hi] + cx.y, hr[4 * lcs + hi] + cx.z};
                epilogue_cell<T, MODE>(r, cell, mi, mi, b, ms, ynv, accv, none, stage, step, wb, ynv, accv);
            }
            __syncthreads();
        }
        if (SEG && !RELAX && rank == 0 && tid == 0 && seg.signal) post_progress(flags + seg.rep, n);
        if (RELAX && conv_s) break;
    }
    // the final state of the CTA's cells back to the caller's buffer
    bool bad = false;
    if (MODE != M_FIELD)
    for (int k = c0 + tid; k < c1; k += NT) {
        const int cell = __ldg(r.cells + k);
        const int y = cell / D, x = cell - y * D;
        const long long mi = (long long)(y - ylo) * Dpad + x;
        const vec3<T> v = RELAX ? ms.ld(mi) : ynv.ld(mi);
        yg.st((long long)y * Dpad + x, v);
        bad |= !finite3(v);
    }
    if (MODE == M_RK4 || MODE == M_HEUN) flag_nan(bad, status);
    if (WIDE && rank == 0 && tid < 2) __stcg(&rx.rio[seg.rep].lam[tid], (double)lam2.hi + (double)lam2.lo);
    if (RELAX && rank == 0 && tid == 0) {
        RelaxIO *io = rx.rio + seg.rep;
        const int iters = __ldcg(&io->iters) + (int)n;
        if (!WIDE) {
            __stcg(&io->lam[0], (double)lam_s[0]);
            __stcg(&io->lam[1], (double)lam_s[1]);
        }
        __stcg(&io->resid, (double)res_last);
        __stcg(&io->iters, iters);
        if (conv_s) __stcg(&io->status, 0);
        if (conv_s || iters >= rx.max_iter) atomicAdd(rx.ndone, 1);
    }
    if (SEG && seg.signal) {   // every CTA's rows are written before the flag
        __threadfence();
        cluster.sync();
        if (rank == 0 && tid == 0) {
            __threadfence();
            if (RELAX) atomicAdd(flags + seg.rep, 1);
            else atomicExch(flags + seg.rep, kHandedOver);
        }
    }
    }
    cluster.sync();   // no CTA leaves while another may still access its shared memory
}

// Launch configuration of one replica per cluster of NC CTAs (the cluster
// shape is a launch attribute; NC = 16 is a non-portable size the GPU allows).
template <int P, typename T, int MODE, int NC, bool SEG>
static cudaError_t cluster_config(cudaLaunchConfig_t &cfg, cudaLaunchAttribute *attr, int nclusters, size_t sm,
                                  cudaStream_t st)
{
    auto kern = k_cluster<P, T, MODE, NC, SEG>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e == cudaSuccess && NC > 8) e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
    cfg = cudaLaunchConfig_t{};
    cfg.gridDim = dim3(nclusters * NC, 1, 1);
    cfg.blockDim = dim3(ClusterGeom<P, T, NC>::NT, 1, 1);
    cfg.dynamicSmemBytes = sm;
    cfg.stream = st;
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = NC;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaSuccess;
}

template <int P, typename T, int MODE, int NC, bool SEG>
static cudaError_t launch_cluster_t(const LaunchArgs &a, int maxD, int maxDpad)
{
    const size_t sm = cluster_smem_bytes<P, T, NC>(maxD, maxDpad, a.use_wbuf != 0);
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr[1];
    cudaError_t e = cluster_config<P, T, MODE, NC, SEG>(cfg, attr, SEG ? a.ncta : a.nwork, sm, a.stream);
    if (e != cudaSuccess) return e;
    const ClusterRelax rx = {a.rio, (const double *)a.tw64, a.eta, a.tol, a.rc2, a.max_iter, a.quantum, a.nwork,
                             a.flags ? a.flags + a.n_rep + 1 : nullptr};
    return cudaLaunchKernelEx(&cfg, k_cluster<P, T, MODE, NC, SEG>, a.reps, a.work, (T *)a.y, (T *)a.out,
                              (const cplx<T> *)a.tw, a.nsteps, a.step_base, a.use_wbuf, a.status, a.segs,
                              a.seg_off, a.flags, a.flags ? a.flags + a.n_rep : nullptr, a.wait_polls, rx);
}

// Clusters of the size class that can be resident at once (0: the cluster
// shape or its shared memory does not fit this GPU).
template <int P, typename T, int NC>
static int cluster_max_active_t(int maxD, int maxDpad, bool wbuf)
{
    const size_t sm = cluster_smem_bytes<P, T, NC>(maxD, maxDpad, wbuf);
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr[1];
    if (cluster_config<P, T, M_HEUN, NC, false>(cfg, attr, 1, sm, 0) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, k_cluster<P, T, M_HEUN, NC, false>, &cfg) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return n;
}

template <int P, typename T, int NC>
static cudaError_t launch_cluster_p(const LaunchArgs &a, int maxD, int maxDpad)
{
    if (a.mode == M_RK4)
        return a.segs ? launch_cluster_t<P, T, M_RK4, NC, true>(a, maxD, maxDpad)
                      : launch_cluster_t<P, T, M_RK4, NC, false>(a, maxD, maxDpad);
    if (a.mode == M_HEUN)
        return a.segs ? launch_cluster_t<P, T, M_HEUN, NC, true>(a, maxD, maxDpad)
                      : launch_cluster_t<P, T, M_HEUN, NC, false>(a, maxD, maxDpad);
    if (a.mode == M_RELAX) return launch_cluster_t<P, T, M_RELAX, NC, true>(a, maxD, maxDpad);
    if (a.mode == M_FIELD) return launch_cluster_t<P, T, M_FIELD, NC, false>(a, maxD, maxDpad);
    return cudaErrorInvalidValue;
}

}  // namespace nd
