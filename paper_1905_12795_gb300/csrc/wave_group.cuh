// The plain streaming and the L2 modelling kernels' common part: an instance on
// a group of co-resident CTAs, its time levels in global memory (L2-resident).
//
// A group of CTAs of WAVE_THREADS threads owns one instance at a time, taken
// from a global queue.  Its two wavefield buffers live in a private slot, with
// few enough groups in flight that the slots and model fields stay in L2.  The
// grid is cut into runs of rows, one run of one float4 column group per thread
// of the whole group (item i = run NQ + column on thread i, so a warp's lanes
// read neighbouring columns).  A thread walks its run with the 2R+1 rows of the
// z-stencil in a register window; the rows of u^n, u^{n-1} and a that it needs
// PF rows later are requested PF rows ahead, which is what hides the L2 latency
// at the 8 to 12 warps per SM that the registers allow.  u^{n+1} overwrites
// u^{n-1} in place.  The CTAs of a group meet once per step at an arrive
// counter in global memory (they are co-resident: cooperative launch); the
// acquire makes the plain, L1-cached loads of the next step see the other SMs'
// stores.  A group may have any number of CTAs, so no SM is left out: clusters
// of 10 CTAs, the best of the thread-block clusters, reach 130 of 152 SMs and
// take 16 instances in two rounds.  Receivers are shared out over the group's
// CTAs; their samples of u^n are copied to shared memory under the sweep.
#pragma once

#include <algorithm>
#include <map>
#include <mutex>

#include "internal.cuh"
#include "stencil.cuh"

namespace empso {

namespace {

constexpr int WAVE_THREADS = 128;
constexpr int PF = 3;                    // rows requested ahead

// A run is swept U rows per pass of the loop, after which its register window
// of N rows moves by U (11 register moves a row at radius 4, 19 at radius 8).  A
// ring unrolled over its whole length needs no moves, but is 50 KB of code at
// either radius, and the warps waited for instructions (2 of 6 to 8 cycles per
// issue, ncu): 44.5 against 33 us a step, order 16, 16 instances on the 1041 x
// 421 grid.
constexpr int U = PF + 1;
template <int R> struct Window {
    static constexpr int N = 2 * R + PF + U;
};

struct Corners {
    int k;          // buffer offset of the lower-left corner
    float w[4];     // (i0,j0) (i0+1,j0) (i0,j0+1) (i0+1,j0+1)
};

__device__ __forceinline__ Corners bilinear(float x, float z, const GridDev &g)
{
    float fx = x / g.hx + (float)g.pad;
    float fz = z / g.hz + (float)g.pad;
    int i0 = (int)floorf(fx), j0 = (int)floorf(fz);
    i0 = min(max(i0, 0), g.NX - 2);
    j0 = min(max(j0, 0), g.NZ - 2);
    float ax = fx - (float)i0, az = fz - (float)j0;
    Corners c;
    c.k = (j0 + HALO) * g.pitch + i0 + HALO;
    c.w[0] = (1.f - ax) * (1.f - az);
    c.w[1] = ax * (1.f - az);
    c.w[2] = (1.f - ax) * az;
    c.w[3] = ax * az;
    return c;
}

constexpr int WS_LINE = 32;              // ints of a line of the launch's workspace

// The step barrier of a group of n CTAs: an arrive counter in global memory that
// thread 0 releases (after the CTA barrier, so for all its threads' stores) and
// polls, with one acquiring fence once everybody is there.  `target` is thread
// 0's running count.  False when the wait gave up (WAIT_LIMIT_NS).  (Fences
// around the release and an acquiring load per poll cost 0.3 us a step; eight
// counters on lines of their own were slower than one.)
__device__ __forceinline__ bool group_barrier(unsigned *count, unsigned &target, int n, int *s_fail)
{
    __syncthreads();
    if (n == 1) return true;
    if (threadIdx.x == 0) {
        target += (unsigned)n;
        asm volatile("red.release.gpu.global.add.u32 [%0], 1;\n" ::"l"(count) : "memory");
        unsigned long long t0 = 0;
        for (unsigned spin = 0;; ++spin) {
            unsigned v;
            asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];\n" : "=r"(v) : "l"(count) : "memory");
            if ((int)(v - target) >= 0) break;
            if ((spin & 255u) == 255u) {
                const unsigned long long t = global_ns();
                if (t0 == 0) t0 = t;
                else if (t - t0 > WAIT_LIMIT_NS) {
                    *s_fail = 1;
                    break;
                }
            }
        }
        asm volatile("fence.acq_rel.gpu;\n" ::: "memory");
    }
    __syncthreads();
    return *s_fail == 0;
}

// A warp's rows of u^n in shared memory, for the x-stencil: XG edge groups
// either side of the 32 lanes' own and one group of zeros; ROWS rows in turn
// (the edges of the next PF rows are on the way while a row is read).
template <int R> struct XRow {
    static constexpr int XG = XGroups<R>::G, ZERO = 32 + 2 * XG, LEN = ZERO + 1, ROWS = U;
    static_assert(ROWS > PF, "a row's edges arrive while the rows before it are read");
};

__device__ __forceinline__ void cp_async4(float *sdst, const float *gsrc)
{
    const unsigned d = (unsigned)__cvta_generic_to_shared(sdst);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(d), "l"(gsrc) : "memory");
}

__device__ __forceinline__ void cp_async16(void *sdst, const void *gsrc)
{
    const unsigned d = (unsigned)__cvta_generic_to_shared(sdst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d), "l"(gsrc) : "memory");
}

// a byte offset into a buffer
template <bool WIDE> struct ByteOffset {
    using type = unsigned;
};
template <> struct ByteOffset<true> {
    using type = unsigned long long;
};

// num / d for 1 <= d < 4096: a reciprocal after one Newton step on the hardware's
// approximation, and the quotient corrected by its remainder (Markstein's method:
// correctly rounded where the remainder is exact, for |num| from 2^-90 up; below, the
// remainder may be subnormal, and the error within half a last place and 2^-150);
// d = 1 returns num, and infinities and not-a-numbers stay what they are (the
// remainder of an infinity is not a number: the larger of it and -MOST is -MOST, and
// its product added to the infinity leaves that).  With the compiler's division in its
// place the damping layer's rows took twice the time of the others (60 cells, order 16,
// 16 instances on the 1041 x 421 grid: 33.6 us a step against 21.6); correctly
// rounded below 2^-90 too, by scaling, those rows cost a fifth more, and the waves'
// first traces, where such numbers are, run ahead of them through the whole grid.
// FINITE: num is known to be.
template <bool FINITE = false>
__device__ __forceinline__ float2 quot2(float2 num, float2 d)
{
    float2 y;
    asm("rcp.approx.ftz.f32 %0, %1;\n" : "=f"(y.x) : "f"(d.x));
    asm("rcp.approx.ftz.f32 %0, %1;\n" : "=f"(y.y) : "f"(d.y));
    const float2 nd = __fmul2_rn(splat2(-1.f), d);
    y = __ffma2_rn(y, __ffma2_rn(nd, y, splat2(1.f)), y);
    const float2 q = __fmul2_rn(num, y);
    float2 r = __ffma2_rn(nd, q, num);
    constexpr float MOST = 0x1.fffffep127f;
    if (!FINITE) r = f2(fmaxf(r.x, -MOST), fmaxf(r.y, -MOST));
    return __ffma2_rn(r, y, q);
}

// One step of one run: rows j0 .. j0 + len - 1 of column group q, the whole
// warp together (lmax: the longest run of the warp, at most one row longer than
// the shortest; the last run of a column is never the shorter, so a lane may
// read one row past its own; `act` false: a lane that only goes along; lanes hold
// consecutive columns, and where the columns wrap to the next run the neighbours
// are the zeros outside the grid).  The x-neighbours come from the other lanes
// through shared memory and, past the warp's ends, from one group that XG lanes
// at each end copy there PF rows ahead: read from global memory in the row that
// needs them they would wait in the L1's order behind the rows just requested.
// Rows whose requests lie inside every lane's run are swept without a test (a
// second copy of the row, 20 KB of code in all; with a test in every row the
// integer operations of a row doubled).
//
// GF false: u^{n+1} = [a lap + (2 u^n - (1 - t) u^{n-1})] / (1 + t), the scheme
// as written.  GF true: u^{n+1} = g (u^n - u^{n-1}) + u^{n-1} + (a g / 2) lap
// with g = 2 / (1 + t), fewer operations and a tenth of the rounding error.
//
// Byte offsets into a buffer are 32 bits wide (64-bit ones cost an addition per
// access: 33 against 31 us a step, order 16, 16 instances on the 1041 x 421 grid).
// WIDE, for buffers of 4 GB and more: 64 bits.
template <int R, bool GF, bool HIST, bool WIDE>
__device__ __forceinline__ void sweep_run(const GridDev &g, const float4 *cur, float4 *prev, float4 *hist,
                                          const float4 *__restrict__ a4, int p4, int q, int j0, int len, bool act,
                                          int lmax, float4 *xb, const float *cx, const float *cz, float cres,
                                          int s_i0, int s_j0, const float *sw, float rn)
{
    constexpr int N = Window<R>::N, XG = XRow<R>::XG, ZERO = XRow<R>::ZERO, LEN = XRow<R>::LEN;
    using Ofs = typename ByteOffset<WIDE>::type;
    const int lane = threadIdx.x & 31, NQ = g.NQ;
    // byte offsets into the buffers: row k's own group, the ones requested in row k,
    // and the edge group
    const Ofs pb = (Ofs)p4 * 16u;
    Ofs o_st = ((Ofs)(j0 + HALO) * (Ofs)p4 + HALO4 + q) * 16u;
    Ofs o_um = o_st + PF * pb, o_w = o_st + (R + PF) * pb;
    unsigned o_ez = (unsigned)(j0 + HALO + PF) * 4u;
    auto ld = [](const char *p, Ofs o) { return *reinterpret_cast<const float4 *>(p + o); };
    auto ldg = [](const char *p, Ofs o) { return __ldg(reinterpret_cast<const float4 *>(p + o)); };
    // the edge group this lane fetches for the warp: the run of lane 0 or 31
    const bool left = lane < XG, edge = left || lane >= 32 - XG;
    const int src = left ? 0 : 31;
    const int qe = __shfl_sync(0xffffffffu, q, src), je = __shfl_sync(0xffffffffu, j0, src);
    Ofs o_e = ((Ofs)(je + HALO) * (Ofs)p4 + HALO4 + qe + (left ? lane - XG : lane - (32 - XG) + 1)) * 16u;
    float4 *eslot = xb + (left ? lane : lane + 2 * XG), *own = xb + XG + lane;
    // where the x-neighbours are
    const float4 *x_l = xb + (q >= 1 ? XG + lane - 1 : ZERO), *x_r = xb + (q + 1 < NQ ? XG + lane + 1 : ZERO);
    const float4 *x_l2 = xb + (q >= 2 ? XG + lane - 2 : ZERO), *x_r2 = xb + (q + 2 < NQ ? XG + lane + 2 : ZERO);
    const float4 ex = __ldg(reinterpret_cast<const float4 *>(g.ex + HALO) + q);
    // some column of the warp in the x-damping layer (the same for all its lanes)
    const bool xpad = __any_sync(0xffffffffu, ex.x != 0.f || ex.y != 0.f || ex.z != 0.f || ex.w != 0.f);
    const float2 gx01 = GF ? f2(2.f / (1.f + ex.x), 2.f / (1.f + ex.y)) : splat2(0.f);
    const float2 gx23 = GF ? f2(2.f / (1.f + ex.z), 2.f / (1.f + ex.w)) : splat2(0.f);
    // the run's row of the source's first corner, when one of the source's
    // columns is in this group
    const int ks = act && s_i0 >= 4 * q - 1 && s_i0 <= 4 * q + 3 ? s_j0 - j0 : -2;
    const bool src_here = ks + 1 >= 0 && ks < len;
    const char *cu = reinterpret_cast<const char *>(cur), *au = reinterpret_cast<const char *>(a4);
    const char *zu = reinterpret_cast<const char *>(g.ez);
    char *pu = reinterpret_cast<char *>(prev), *hu = reinterpret_cast<char *>(hist);
    float4 w[N], um[U], av[U];
    float ez[U];
#pragma unroll
    for (int m = 0; m < 2 * R + PF; ++m)
        if (m - 2 * R < lmax) w[m] = ld(cu, o_st + (m - R) * pb);
#pragma unroll
    for (int m = 0; m < PF; ++m) {
        if (m < lmax) {
            um[m] = ld(pu, o_st + m * pb);
            av[m] = ldg(au, o_st + m * pb);
            ez[m] = __ldg(g.ez + j0 + HALO + m);
            if (edge) cp_async16(eslot + m * LEN, cu + o_e + m * pb);
        }
        asm volatile("cp.async.commit_group;\n" ::: "memory");
    }
    o_e += PF * pb;
    // row k = k0 + kk of the run: requests what row k + PF needs; full: there is
    // such a row in every lane's run
    auto row = [&](const int k0, const int kk, const bool full) {
        const int k = k0 + kk, s = kk * LEN, kn = (kk + PF) % U;
        const float4 *wl = w + kk;
        own[s] = wl[R];
        asm volatile("cp.async.wait_group %0;\n" ::"n"(PF - 1) : "memory");
        __syncwarp();
        if (full || k + PF < lmax) {
            w[kk + 2 * R + PF] = ld(cu, o_w);
            um[kn] = ld(pu, o_um);
            av[kn] = ldg(au, o_um);
            ez[kn] = __ldg(reinterpret_cast<const float *>(zu + o_ez));
            if (edge) cp_async16(eslot + kn * LEN, cu + o_e);
        }
        asm volatile("cp.async.commit_group;\n" ::: "memory");
        float xs[4 * (2 * XG + 1)];
        if (XG == 1) xline1(x_l[s], wl[R], x_r[s], xs);
        else xline2(x_l2[s], x_l[s], wl[R], x_r[s], x_r2[s], xs);
        float2 l01, l23;
        lap_group<R>(wl, xs, cx, cz, cres, l01, l23);
        // the gradient's history: L u^n without the source term (written once: evict first)
        if (HIST && act && (full || k < len))
            __stcs(reinterpret_cast<float4 *>(hu + o_st), make_float4(l01.x, l01.y, l23.x, l23.y));
        if (src_here && (k == ks || k == ks + 1)) {
            const float w0 = k == ks ? sw[0] : sw[2], w1 = k == ks ? sw[1] : sw[3];
            float lv[4] = {l01.x, l01.y, l23.x, l23.y};
#pragma unroll
            for (int l = 0; l < 4; ++l) {
                const int I = 4 * q + l;
                lv[l] = fmaf((I == s_i0 ? w0 : 0.f) + (I == s_i0 + 1 ? w1 : 0.f), rn, lv[l]);
            }
            l01 = f2(lv[0], lv[1]);
            l23 = f2(lv[2], lv[3]);
        }
        const float4 u0 = um[kk], a0 = av[kk];
        const float2 mone = splat2(-1.f);
        float2 n01, n23;
        if (GF) {
            float2 g01 = gx01, g23 = gx23;
            if (ez[kk] != 0.f) {
                g01 = f2(__fdividef(2.f, 1.f + (ex.x + ez[kk])), __fdividef(2.f, 1.f + (ex.y + ez[kk])));
                g23 = f2(__fdividef(2.f, 1.f + (ex.z + ez[kk])), __fdividef(2.f, 1.f + (ex.w + ez[kk])));
            }
            const float2 half = splat2(0.5f);
            const float2 af01 = __fmul2_rn(lo2(a0), __fmul2_rn(g01, half)), af23 = __fmul2_rn(hi2(a0), __fmul2_rn(g23, half));
            n01 = __ffma2_rn(g01, __ffma2_rn(lo2(u0), mone, lo2(wl[R])), __ffma2_rn(af01, l01, lo2(u0)));
            n23 = __ffma2_rn(g23, __ffma2_rn(hi2(u0), mone, hi2(wl[R])), __ffma2_rn(af23, l23, hi2(u0)));
        } else if (ez[kk] != 0.f || xpad) {
            const float2 two = splat2(2.f), z = splat2(ez[kk]), one = splat2(1.f);
            const float2 t01 = __fadd2_rn(lo2(ex), z), t23 = __fadd2_rn(hi2(ex), z);
            n01 = __fmul2_rn(__fadd2_rn(t01, mone), lo2(u0));         // -(1 - t) u^{n-1}
            n23 = __fmul2_rn(__fadd2_rn(t23, mone), hi2(u0));
            n01 = __ffma2_rn(lo2(a0), l01, __ffma2_rn(two, lo2(wl[R]), n01));
            n23 = __ffma2_rn(hi2(a0), l23, __ffma2_rn(two, hi2(wl[R]), n23));
            n01 = quot2(n01, __fadd2_rn(t01, one));
            n23 = quot2(n23, __fadd2_rn(t23, one));
        } else {
            n01 = __ffma2_rn(lo2(a0), l01, __ffma2_rn(mone, lo2(u0), __fadd2_rn(lo2(wl[R]), lo2(wl[R]))));
            n23 = __ffma2_rn(hi2(a0), l23, __ffma2_rn(mone, hi2(u0), __fadd2_rn(hi2(wl[R]), hi2(wl[R]))));
        }
        if (act && (full || k < len)) *reinterpret_cast<float4 *>(pu + o_st) = make_float4(n01.x, n01.y, n23.x, n23.y);
        o_st += pb;
        o_um += pb;
        o_w += pb;
        o_e += pb;
        o_ez += 4u;
    };
    int k0 = 0;
    for (; k0 + U - 1 + PF < lmax; k0 += U) {
#pragma unroll
        for (int kk = 0; kk < U; ++kk) row(k0, kk, true);
#pragma unroll
        for (int m = 0; m < N - U; ++m) w[m] = w[m + U];
    }
    for (; k0 < lmax; k0 += U) {
#pragma unroll
        for (int kk = 0; kk < U; ++kk)
            if (k0 + kk < lmax) row(k0, kk, false);
#pragma unroll
        for (int m = 0; m < N - U; ++m) w[m] = w[m + U];
    }
    asm volatile("cp.async.wait_group 0;\n" ::: "memory");
}

// CTA `rank` of a group of n runs its part of instance `in`; bufA / bufB are
// the group's slot.  False when a barrier gave up.
template <int R, bool GF, bool HIST, bool WIDE>
__device__ bool run_instance(const GridDev &g, const Inst &in, float *bufA, float *bufB, float4 *xrows,
                             float (*samples)[WAVE_THREADS], int rank, int n, unsigned *count, unsigned &target,
                             int *s_fail, double *red, double *gpart, double *partial)
{
    const int tid = threadIdx.x, nth = n * WAVE_THREADS, gt = rank * WAVE_THREADS + tid, lane = tid & 31;
    float4 *xb = xrows + (tid >> 5) * XRow<R>::ROWS * XRow<R>::LEN;
    if (lane < XRow<R>::ROWS) xb[lane * XRow<R>::LEN + XRow<R>::ZERO] = make_float4(0.f, 0.f, 0.f, 0.f);
    // zero both time levels (interior, halo and alignment columns; bufB follows bufA)
    {
        float4 *z4 = reinterpret_cast<float4 *>(bufA);
        const long long n4 = (2 * g.field) / 4;
        for (long long e = gt; e < n4; e += nth) z4[e] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    // source corners and per-node weights b / (hx hz)
    const Corners sc = bilinear(in.sx, in.sz, g);
    const int s_j0 = sc.k / g.pitch - HALO, s_i0 = sc.k % g.pitch - HALO;
    const float inv_cell = 1.f / (g.hx * g.hz);
    // (the two forms place the source term's cell area differently)
    const float w_cell = GF ? inv_cell : 1.f, r_cell = GF ? 1.f : inv_cell;
    const float sw[4] = {sc.w[0] * w_cell, sc.w[1] * w_cell, sc.w[2] * w_cell, sc.w[3] * w_cell};
    const int NQ = g.NQ, p4 = g.pitch / 4;
    const int nseg = max(1, min(g.NZ, nth / NQ)), items = NQ * nseg;
    const float4 *a4 = reinterpret_cast<const float4 *>(in.a);

    float cx[R + 1], cz[R + 1];
#pragma unroll
    for (int m = 0; m <= R; ++m) {
        cx[m] = g.cxm[m];
        cz[m] = g.czm[m];
    }
    const float cres = g.cres;
    const int rec_b = (int)((long long)rank * in.nrec / n), rec_e = (int)((long long)(rank + 1) * in.nrec / n);
    // a thread's first receiver: its corner and weights; its four samples and
    // its observed value are copied to shared memory while the step is swept
    const int r0 = rec_b + tid;
    const bool has_rec = r0 < rec_e;
    Corners rc{};
    if (has_rec) rc = bilinear(in.rec[r0].x, in.rec[r0].y, g);
    // The residual energy.  GF false: each square is formed and added in FP64.  GF
    // true: 32 squares are added in FP32, as the on-chip kernel does, then carried in
    // FP64: 32 steps of a thread with one receiver, fewer where a thread has more
    // (groups of few CTAs).  (FP64 sums for a thread's further receivers, in this loop:
    // 0.5 to 3 % on the 921 x 301 grid, whose threads have none.)
    const int per = (rec_e - rec_b + WAVE_THREADS - 1) / WAVE_THREADS;    // receivers of a thread
    const int flush = per <= 1 ? 31 : (per <= 2 ? 15 : (per <= 4 ? 7 : (per <= 8 ? 3 : (per <= 16 ? 1 : 0))));
    float accf = 0.f;
    double acc = 0.0;
    auto record = [&](int r, int step, float d, float obs) {
        if (in.traces) in.traces[(size_t)(step - 1) * in.nrec + r] = d;
        if (in.dobs) {
            const float e = d - obs;
            if (GF) accf = fmaf(e, e, accf);
            else acc += (double)e * (double)e;
        }
    };
    if (!group_barrier(count, target, n, s_fail)) return false;

    float *cur = bufA, *prev = bufB;
    for (int step = 0; step <= g.nt; ++step) {
        // receivers sample u^n (record n - 1): `cur` is read-only this step
        if (step >= 1 && has_rec) {
            cp_async4(&samples[0][tid], cur + rc.k);
            cp_async4(&samples[1][tid], cur + rc.k + 1);
            cp_async4(&samples[2][tid], cur + rc.k + g.pitch);
            cp_async4(&samples[3][tid], cur + rc.k + g.pitch + 1);
            if (in.dobs) cp_async4(&samples[4][tid], in.dobs + (size_t)(step - 1) * in.nrec + r0);
        }
        for (int r = r0 + WAVE_THREADS; step >= 1 && r < rec_e; r += WAVE_THREADS) {
            const Corners c = bilinear(in.rec[r].x, in.rec[r].y, g);
            const float d = c.w[0] * cur[c.k] + c.w[1] * cur[c.k + 1] +
                            c.w[2] * cur[c.k + g.pitch] + c.w[3] * cur[c.k + g.pitch + 1];
            record(r, step, d, in.dobs ? in.dobs[(size_t)(step - 1) * in.nrec + r] : 0.f);
        }
        const float rn = step < g.nt ? g.wavelet[step] * r_cell : 0.f;
        for (int i0 = gt - lane; step < g.nt && i0 < items; i0 += nth) {      // a warp at a time
            const int item = i0 + lane;
            const bool act = item < items;                     // lanes past the end go along with the last run
            const int q = min(item, items - 1) % NQ, seg = min(item, items - 1) / NQ;
            const int j0 = (int)((long long)seg * g.NZ / nseg), j1 = (int)((long long)(seg + 1) * g.NZ / nseg);
            const int len = j1 - j0;
            sweep_run<R, GF, HIST, WIDE>(g, reinterpret_cast<const float4 *>(cur), reinterpret_cast<float4 *>(prev),
                         HIST ? reinterpret_cast<float4 *>(in.hist + (size_t)(step + 1) * g.field) : nullptr, a4, p4,
                         q, j0, len, act, __reduce_max_sync(0xffffffffu, len), xb, cx,
                         cz, cres, s_i0, s_j0, sw, rn);
            __syncwarp();                                      // the last rows' reads, before the next run's
        }
        if (step >= 1 && has_rec) {
            asm volatile("cp.async.wait_all;\n" ::: "memory");
            record(r0, step,
                   rc.w[0] * samples[0][tid] + rc.w[1] * samples[1][tid] + rc.w[2] * samples[2][tid] +
                       rc.w[3] * samples[3][tid],
                   in.dobs ? samples[4][tid] : 0.f);
        }
        if (GF && (step & flush) == 0) {
            acc += (double)accf;
            accf = 0.f;
        }
        if (step == g.nt) break;
        if (!group_barrier(count, target, n, s_fail)) return false;
        float *t = cur;
        cur = prev;
        prev = t;
    }
    acc += (double)accf;
    // fixed-order reduction of the residual energy: warps, CTA, group
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
    if ((tid & 31) == 0) red[tid >> 5] = acc;
    __syncthreads();
    if (tid == 0) {
        double v = 0.0;
        for (int w = 0; w < WAVE_THREADS / 32; ++w) v += red[w];
        gpart[rank] = v;
    }
    if (!group_barrier(count, target, n, s_fail)) return false;
    if (rank == 0 && tid == 0) {
        double v = 0.0;
        for (int c = 0; c < n; ++c) v += __ldcg(gpart + c);
        partial[in.out] = 0.5 * v;
    }
    return true;
}

// The launch's workspace: line 0 the instance queue, then one 128-byte line
// per group (arrive count, the group's instance), then one partial misfit per
// CTA (wave_ws_bytes holds any split).

template <int R> struct Radius {
    static constexpr int value = R;
};

// CTAs per SM that the registers are held to
template <int RF> struct GroupCtas {
    static constexpr int v = RF == 0 || RF == 8 ? 2 : 3;
};

// a CTA's whole work; RF: the radius of every grid of the launch (0: per instance);
// WIDE: some grid's buffer holds 4 GB or more
template <int RF, bool GF, bool HIST, bool WIDE>
__device__ __forceinline__ void group_cta(const GridDev *__restrict__ grids, const Inst *__restrict__ insts, int n_inst,
                                          int group, int *ws, float *slots, long long slot_floats, int *err,
                                          double *partial)
{
    __shared__ float4 xrows[WAVE_THREADS / 32 * U * XRow<RF ? RF : MAX_R>::LEN];
    __shared__ float samples[5][WAVE_THREADS];
    __shared__ double red[WAVE_THREADS / 32];
    __shared__ GridDev sg;
    __shared__ int s_q, s_fail;
    const int gid = blockIdx.x / group, rank = blockIdx.x % group, groups = gridDim.x / group;
    int *line = ws + WS_LINE * (1 + gid);
    unsigned *count = reinterpret_cast<unsigned *>(line);
    double *gpart = reinterpret_cast<double *>(ws + WS_LINE * (1 + groups)) + (size_t)gid * group;
    float *bufA = slots + (size_t)gid * slot_floats;
    unsigned target = 0;
    if (threadIdx.x == 0) s_fail = 0;
    for (;;) {
        if (rank == 0 && threadIdx.x == 0) {
            const int q = atomicAdd(ws, 1);
            __stcg(line + 1, q);
            // a group that gives up leaves its instance's misfit not a number
            if (q < n_inst) partial[insts[q].out] = __longlong_as_double(0x7ff8000000000000LL);
        }
        if (!group_barrier(count, target, group, &s_fail)) break;
        if (threadIdx.x == 0) s_q = __ldcg(line + 1);
        __syncthreads();
        const int q = s_q;
        if (q >= n_inst) break;
        const Inst in = insts[q];
        if (threadIdx.x == 0) sg = grids[in.grid];
        __syncthreads();
        const GridDev &g = sg;
        float *bufB = bufA + g.field;
        auto run = [&](auto r) {
            return run_instance<decltype(r)::value, GF, HIST, WIDE>(g, in, bufA, bufB, xrows, samples, rank, group, count,
                                                             target, &s_fail, red, gpart, partial);
        };
        bool ok;
        if constexpr (RF != 0) ok = run(Radius<RF>{});
        else if (!GF && g.R == 8) ok = run(Radius<GF ? 4 : 8>{});     // (GF: the L2 kernel, radius up to 4)
        else if (g.R == 4) ok = run(Radius<4>{});
        else if (g.R == 2) ok = run(Radius<2>{});
        else ok = run(Radius<1>{});
        if (!ok) break;
    }
    if (threadIdx.x == 0 && s_fail) {
        // a group that gave up also takes what is left of the queue: no instance keeps
        // what an earlier launch left as its misfit
        if (rank == 0)
            for (int q = atomicAdd(ws, 1); q < n_inst; q = atomicAdd(ws, 1))
                partial[insts[q].out] = __longlong_as_double(0x7ff8000000000000LL);
        if (err) atomicExch(err, EMPSO_TIMEOUT);
    }
}

using WaveFn = void (*)(const GridDev *, const Inst *, int, int, int *, float *, long long, int *, double *);

// co-resident CTAs of a group kernel on the current device (memoised)
inline int group_max_ctas(WaveFn fn)
{
    static std::mutex mu;
    static std::map<std::pair<int, WaveFn>, int> memo;
    int dev = 0, sms = 0, n = 0;
    if (!fn || cudaGetDevice(&dev) != cudaSuccess) return 0;
    std::lock_guard<std::mutex> lock(mu);
    const auto it = memo.find({dev, fn});
    if (it != memo.end()) return it->second;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, fn, WAVE_THREADS, 0) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return memo[{dev, fn}] = std::min(sms * n, WAVE_MAX_CTAS);
}

// does some grid's buffer need 64-bit byte offsets?
inline bool group_wide(const GridDev *const *grids, int n_grids)
{
    bool wide = false;
    for (int i = 0; i < n_grids; ++i) wide = wide || 4 * grids[i]->field > 1LL << 32;
    return wide;
}

// Instances in flight and CTAs per instance: the split of the co-resident CTAs
// with the least estimated time, rounds of instances x rows a thread sweeps
// (plus RUN_EXTRA rows' worth for the window it loads first and the step
// barrier, of which RUN_BARRIER for the barrier, which one CTA does without), with
// at most `by_l2` instances in flight; `fixed` > 0: so many CTAs per instance.  The
// barrier is 1.2 us a step on a GPU of few groups and 1.8 on one of many, a row 0.24:
// order 8, 103 steps, 1 and 64 models of 21 x 21 + 4 cells 347 and 403 us on groups
// of 2 CTAs, 258 and 263 on one CTA each; 41 x 31 + 8 cells 366 and 453, 351 and 363;
// 61 x 41 + 10 cells 402 and 495 on 8 and 4 CTAs, 474 and 504.
inline WaveSplit group_split(const GridDev *const *grids, int n_grids, int ctas, long long n_inst, long long by_l2,
                             int fixed = 0)
{
    constexpr int RUN_EXTRA = 10, RUN_BARRIER = 6;
    WaveSplit best{};
    best.wide = group_wide(grids, n_grids);
    const long long most = std::max<long long>(1, std::min<long long>({n_inst, by_l2, (long long)ctas}));
    double cost = 0.0;
    if (ctas > 0 && fixed > 0) {
        best.group = std::min(fixed, ctas);
        best.flight = (int)std::min<long long>(most, ctas / best.group);
        return best;
    }
    for (long long f = 1; f <= most && ctas > 0; ++f)
        for (const int n : {(int)(ctas / f), 1}) {       // all the CTAs, or one without a barrier
            long long rows = 0;
            int used = 1;                                // CTAs that have a run to sweep
            for (int i = 0; i < n_grids; ++i) {
                const GridDev &g = *grids[i];
                const int nth = n * WAVE_THREADS, nseg = std::max(1, std::min(g.NZ, nth / g.NQ));
                rows = std::max<long long>(rows, (long long)((g.NZ + nseg - 1) / nseg) * ((g.NQ * nseg + nth - 1) / nth));
                used = std::max(used, std::min(n, (g.NQ * nseg + WAVE_THREADS - 1) / WAVE_THREADS));
            }
            const double c = (double)((n_inst + f - 1) / f) * (double)(rows + RUN_EXTRA - (used == 1 ? RUN_BARRIER : 0));
            if (best.group == 0 || c < cost) {
                cost = c;
                best.flight = (int)f;
                best.group = used;
            }
        }
    return best;
}

inline cudaError_t launch_groups(WaveFn fn, const GridDev *grids_dev, const Inst *insts, int n_inst, const WaveSplit &s,
                                 void *ws, float *slots, long long slot_floats, int *err, double *partial,
                                 cudaStream_t st)
{
    if (n_inst <= 0) return cudaSuccess;
    cudaError_t e = cudaMemsetAsync(ws, 0, sizeof(int) * WS_LINE * (1 + (size_t)s.flight), st);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.gridDim = dim3(s.flight * s.group, 1, 1);
    cfg.blockDim = dim3(WAVE_THREADS, 1, 1);
    cfg.stream = st;
    cfg.attrs = attr;
    cfg.numAttrs = s.group > 1 ? 1 : 0;   // one CTA per instance waits for nobody
    return cudaLaunchKernelEx(&cfg, fn, grids_dev, insts, n_inst, s.group, (int *)ws, slots, slot_floats, err, partial);
}

}  // namespace

}  // namespace empso
