// Acoustic forward modelling of every (model, shot) instance of a generation
// in one persistent launch, with the L2 misfit fused into the time loop
// (section "Testing approach": 2nd order in time, 8th (or 4th) order in space,
// damping layer, Ricker source, receivers along a line, l2 misfit).
//
// Scheme (centred in time, damped, constant density):
//   u^{n+1} = [2 u^n - (1 - t) u^{n-1} + a (lap_h u^n + s^n)] / (1 + t)
// with a = v^2 dt^2, t = (eta_x + eta_z) dt / 2, lap_h the order-2R centred
// Laplacian with zero values outside the padded grid, and s^n the bilinear
// point source r(n dt) b / (hx hz).  Trace sample n is the bilinear sample of
// u^{n+1}; phi = 1/2 sum (d - d_obs)^2.
//
// Work decomposition: a group of CTAs of WAVE_THREADS threads (two per SM)
// owns one instance at a time, taken from a global queue.  Its two wavefield
// buffers live in a private slot of global memory, with few enough groups in
// flight that the slots and model fields stay in L2.  The grid is cut into
// runs of rows, one run of one float4 column group per thread of the whole
// group (item i = run NQ + column on thread i, so a warp's lanes read
// neighbouring columns).  A thread walks its run with the 2R+1 rows of the
// z-stencil in a register ring; the rows of u^n, u^{n-1} and a that it needs
// PF rows later are requested PF rows ahead, which is what hides the L2
// latency at the 8 warps per SM that 255 registers allow, and the ring's
// length is the unroll length, so the window never moves between registers.
// u^{n+1} overwrites u^{n-1} in place.  The CTAs of a group meet once per step
// at an arrive counter in global memory (they are co-resident: cooperative
// launch); the acquire makes the plain, L1-cached loads of the next step see
// the other SMs' stores.  Receivers are shared out over the group's CTAs and
// sample u^n at the start of step n.
//
// Bound by the issue slots (41 % active with 8 warps per SM: the window's 17
// rows leave registers for no more) and the barrier.  Measured, order 16, 16
// shots of the 921 x 301 grid + 60 cells, 2014 steps: 1628 ms with one
// 512-thread CTA per instance (16 SMs busy), 43.1 ms on 16 groups of 19 CTAs
// (327 G updates/s).
#include <algorithm>
#include <map>
#include <mutex>
#include <tuple>

#include "internal.cuh"
#include "stencil.cuh"

namespace empso {

namespace {

constexpr int WAVE_THREADS = 128;
constexpr int PF = 3;                    // rows requested ahead

// A run is swept U rows per pass of the loop; the window then moves by U rows
// (19 register moves a row at radius 8).  A ring unrolled over its whole length
// needs no moves, but at radius 8 that is 50 KB of code and the warps waited
// for instructions (2.8 of 8 cycles per issue, ncu): 44.5 us a step against
// 33 us with U = 4, on the batch above.
constexpr int U = 4;
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

// The step barrier of a group of n CTAs: arrive counter in global memory,
// release by the arriving thread, acquire by the waiting one.  `target` is
// thread 0's running count.  False when the wait gave up (WAIT_LIMIT_NS).
__device__ __forceinline__ bool group_barrier(unsigned *count, unsigned &target, int n, int *s_fail)
{
    __syncthreads();
    if (n == 1) return true;
    if (threadIdx.x == 0) {
        target += (unsigned)n;
        __threadfence();
        asm volatile("red.release.gpu.global.add.u32 [%0], 1;\n" ::"l"(count) : "memory");
        unsigned long long t0 = 0;
        for (unsigned spin = 0;; ++spin) {
            unsigned v;
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];\n" : "=r"(v) : "l"(count) : "memory");
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
        __threadfence();
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

__device__ __forceinline__ void cp_async16(void *sdst, const void *gsrc)
{
    const unsigned d = (unsigned)__cvta_generic_to_shared(sdst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d), "l"(gsrc) : "memory");
}

// num / d for d >= 1: a reciprocal after one Newton step on the hardware's
// approximation, and the quotient corrected by its exact remainder (Markstein's
// method, which gives the correctly rounded quotient); d = 1 returns num.
// With the library's division and reciprocal in their place the damping layer's
// rows took twice the time of the others (60 cells: 33.6 us a step against 21.6)
__device__ __forceinline__ float2 quot2(float2 num, float2 d)
{
    float2 y;
    asm("rcp.approx.ftz.f32 %0, %1;\n" : "=f"(y.x) : "f"(d.x));
    asm("rcp.approx.ftz.f32 %0, %1;\n" : "=f"(y.y) : "f"(d.y));
    const float2 nd = __fmul2_rn(splat2(-1.f), d);
    y = __ffma2_rn(y, __ffma2_rn(nd, y, splat2(1.f)), y);
    const float2 q = __fmul2_rn(num, y);
    return __ffma2_rn(__ffma2_rn(nd, q, num), y, q);
}

// One step of one run: rows j0 .. j0 + len - 1 of column group q, the whole
// warp together (lmin / lmax: the shortest and longest run of the warp; `act`
// false: a lane that only goes along; lanes hold consecutive columns, and where
// the columns wrap to the next run the neighbours are the zeros outside the
// grid).  The x-neighbours come from the other lanes through shared memory and,
// past the warp's ends, from one group that XG lanes at each end copy there PF
// rows ahead: read from global memory in the row that needs them they would
// wait in the L1's order behind the rows just requested.
template <int R, bool HIST>
__device__ __forceinline__ void sweep_run(const GridDev &g, const float4 *cur, float4 *prev, float4 *hist,
                                          const float4 *__restrict__ a4, int p4, int q, int j0, int len, bool act,
                                          int lmin, int lmax, float4 *xb, const float *cx, const float *cz,
                                          float cres, int s_i0, int s_j0, const float *sw, float rn)
{
    constexpr int N = Window<R>::N, UM = PF + 1, XG = XRow<R>::XG, ZERO = XRow<R>::ZERO, LEN = XRow<R>::LEN,
                  ROWS = XRow<R>::ROWS;
    static_assert(UM == U, "a pass of the loop turns the rings once");
    const int lane = threadIdx.x & 31, NQ = g.NQ;
    // byte offsets into the buffers (a buffer holds less than 4 GB): row k's own
    // group, the ones requested in row k, and the edge group
    const unsigned pb = (unsigned)p4 * 16u;
    unsigned o_st = ((unsigned)(j0 + HALO) * (unsigned)p4 + HALO4 + q) * 16u;
    unsigned o_um = o_st + PF * pb, o_w = o_st + (R + PF) * pb, o_ez = (unsigned)(j0 + HALO + PF) * 4u;
    const char *curb = reinterpret_cast<const char *>(cur), *ab = reinterpret_cast<const char *>(a4);
    char *prevb = reinterpret_cast<char *>(prev);
    const char *ezb = reinterpret_cast<const char *>(g.ez);
    auto ld = [](const char *p, unsigned o) { return *reinterpret_cast<const float4 *>(p + o); };
    auto ldg = [](const char *p, unsigned o) { return __ldg(reinterpret_cast<const float4 *>(p + o)); };
    // the edge group this lane fetches for the warp: the run of lane 0 or 31
    const bool left = lane < XG, edge = left || lane >= 32 - XG;
    const int src = left ? 0 : 31;
    const int qe = __shfl_sync(0xffffffffu, q, src), je = __shfl_sync(0xffffffffu, j0, src);
    const int elen = __shfl_sync(0xffffffffu, len, src);
    unsigned o_e = ((unsigned)(je + HALO) * (unsigned)p4 + HALO4 + qe + (left ? lane - XG : lane - (32 - XG) + 1)) * 16u;
    float4 *eslot = xb + (left ? lane : lane + 2 * XG), *own = xb + XG + lane;
    // where the x-neighbours are
    const float4 *x_l = xb + (q >= 1 ? XG + lane - 1 : ZERO), *x_r = xb + (q + 1 < NQ ? XG + lane + 1 : ZERO);
    const float4 *x_l2 = xb + (q >= 2 ? XG + lane - 2 : ZERO), *x_r2 = xb + (q + 2 < NQ ? XG + lane + 2 : ZERO);
    const float4 ex = __ldg(reinterpret_cast<const float4 *>(g.ex + HALO) + q);
    // some column of the warp in the x-damping layer (the same for all its lanes)
    const bool xpad = __any_sync(0xffffffffu, ex.x != 0.f || ex.y != 0.f || ex.z != 0.f || ex.w != 0.f);
    const bool src_here = act && s_i0 >= 4 * q - 1 && s_i0 <= 4 * q + 3 && s_j0 + 1 >= j0 && s_j0 < j0 + len;
    float4 w[N], um[UM], av[UM];
    float ez[UM];
#pragma unroll
    for (int m = 0; m < 2 * R + PF; ++m)
        if (m - 2 * R < len) w[m] = ld(curb, o_st + (m - R) * pb);
#pragma unroll
    for (int m = 0; m < PF; ++m) {
        if (m < len) {
            um[m] = ld(prevb, o_st + m * pb);
            av[m] = ldg(ab, o_st + m * pb);
            ez[m] = __ldg(g.ez + j0 + HALO + m);
        }
        if (edge && m < elen) cp_async16(eslot + m * LEN, curb + o_e + m * pb);
        asm volatile("cp.async.commit_group;\n" ::: "memory");
    }
    o_e += PF * pb;
    // row k = k0 + kk of the run (k0 a multiple of U): requests what row k + PF
    // needs; full: every lane's run goes on past row k + PF
    auto row = [&](const int k0, const int kk, const bool full) {
        const int k = k0 + kk, s = kk * LEN, se = (kk + PF) % ROWS * LEN;
        const float4 *wl = w + kk;
        own[s] = wl[R];
        asm volatile("cp.async.wait_group %0;\n" ::"n"(PF - 1) : "memory");
        __syncwarp();
        if (full || k + PF < len) {
            w[kk + 2 * R + PF] = ld(curb, o_w);
            um[(kk + PF) % UM] = ld(prevb, o_um);
            av[(kk + PF) % UM] = ldg(ab, o_um);
            ez[(kk + PF) % UM] = __ldg(reinterpret_cast<const float *>(ezb + o_ez));
        }
        if (edge && (full || k + PF < elen)) cp_async16(eslot + se, curb + o_e);
        asm volatile("cp.async.commit_group;\n" ::: "memory");
        float xs[4 * (2 * XG + 1)];
        if (XG == 1) xline1(x_l[s], wl[R], x_r[s], xs);
        else xline2(x_l2[s], x_l[s], wl[R], x_r[s], x_r2[s], xs);
        float2 l01, l23;
        lap_group<R>(wl, xs, cx, cz, cres, l01, l23);
        // the gradient's history: L u^n without the source term (written once: evict first)
        if (HIST && act && (full || k < len))
            __stcs(reinterpret_cast<float4 *>(reinterpret_cast<char *>(hist) + o_st), make_float4(l01.x, l01.y, l23.x, l23.y));
        if (src_here) {
            const int j = j0 + k;
            if (j == s_j0 || j == s_j0 + 1) {
                const float w0 = j == s_j0 ? sw[0] : sw[2], w1 = j == s_j0 ? sw[1] : sw[3];
                float lv[4] = {l01.x, l01.y, l23.x, l23.y};
#pragma unroll
                for (int l = 0; l < 4; ++l) {
                    const int I = 4 * q + l;
                    lv[l] = fmaf((I == s_i0 ? w0 : 0.f) + (I == s_i0 + 1 ? w1 : 0.f), rn, lv[l]);
                }
                l01 = f2(lv[0], lv[1]);
                l23 = f2(lv[2], lv[3]);
            }
        }
        // num = a lap + (2 u^n - (1 - t) u^{n-1}), u^{n+1} = num / (1 + t)
        const float4 u0 = um[kk], a0 = av[kk];
        const float2 two = splat2(2.f);
        float2 n01, n23;
        if (ez[kk] != 0.f || xpad) {
            const float2 z = splat2(ez[kk]), one = splat2(1.f), mone = splat2(-1.f);
            const float2 t01 = __fadd2_rn(lo2(ex), z), t23 = __fadd2_rn(hi2(ex), z);
            n01 = __fmul2_rn(__fadd2_rn(t01, mone), lo2(u0));         // -(1 - t) u^{n-1}
            n23 = __fmul2_rn(__fadd2_rn(t23, mone), hi2(u0));
            n01 = __ffma2_rn(lo2(a0), l01, __ffma2_rn(two, lo2(wl[R]), n01));
            n23 = __ffma2_rn(hi2(a0), l23, __ffma2_rn(two, hi2(wl[R]), n23));
            n01 = quot2(n01, __fadd2_rn(t01, one));
            n23 = quot2(n23, __fadd2_rn(t23, one));
        } else {
            const float2 m1 = splat2(-1.f);
            n01 = __ffma2_rn(lo2(a0), l01, __ffma2_rn(m1, lo2(u0), __fadd2_rn(lo2(wl[R]), lo2(wl[R]))));
            n23 = __ffma2_rn(hi2(a0), l23, __ffma2_rn(m1, hi2(u0), __fadd2_rn(hi2(wl[R]), hi2(wl[R]))));
        }
        if (act && (full || k < len)) *reinterpret_cast<float4 *>(prevb + o_st) = make_float4(n01.x, n01.y, n23.x, n23.y);
        o_st += pb;
        o_um += pb;
        o_w += pb;
        o_e += pb;
        o_ez += 4u;
    };
    int k0 = 0;
    for (; k0 + U - 1 + PF < lmin; k0 += U) {
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
template <int R, bool HIST>
__device__ bool run_instance(const GridDev &g, const Inst &in, float *bufA, float *bufB, float4 *xrows, int rank,
                             int n,
                             unsigned *count, unsigned &target, int *s_fail, double *red, double *gpart,
                             double *partial)
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
    double acc = 0.0;
    if (!group_barrier(count, target, n, s_fail)) return false;

    float *cur = bufA, *prev = bufB;
    for (int step = 0; step <= g.nt; ++step) {
        // receivers sample u^n (record n - 1): `cur` is read-only this step
        if (step >= 1) {
            for (int r = rec_b + tid; r < rec_e; r += WAVE_THREADS) {
                const float2 p = in.rec[r];
                const Corners c = bilinear(p.x, p.y, g);
                const float d = c.w[0] * cur[c.k] + c.w[1] * cur[c.k + 1] +
                                c.w[2] * cur[c.k + g.pitch] + c.w[3] * cur[c.k + g.pitch + 1];
                const size_t o = (size_t)(step - 1) * in.nrec + r;
                if (in.traces) in.traces[o] = d;
                if (in.dobs) {
                    const float e = d - in.dobs[o];
                    acc += (double)e * (double)e;
                }
            }
        }
        if (step == g.nt) break;
        const float rn = g.wavelet[step] * inv_cell;
        for (int i0 = gt - lane; i0 < items; i0 += nth) {      // a warp at a time
            const int item = i0 + lane;
            const bool act = item < items;                     // lanes past the end go along with the last run
            const int q = min(item, items - 1) % NQ, seg = min(item, items - 1) / NQ;
            const int j0 = (int)((long long)seg * g.NZ / nseg), j1 = (int)((long long)(seg + 1) * g.NZ / nseg);
            const int len = j1 - j0;
            sweep_run<R, HIST>(g, reinterpret_cast<const float4 *>(cur), reinterpret_cast<float4 *>(prev),
                         HIST ? reinterpret_cast<float4 *>(in.hist + (size_t)(step + 1) * g.field) : nullptr, a4, p4,
                         q, j0, len, act, __reduce_min_sync(0xffffffffu, len), __reduce_max_sync(0xffffffffu, len), xb, cx,
                         cz, cres, s_i0, s_j0, sc.w, rn);
            __syncwarp();                                      // the last rows' reads, before the next run's
        }
        if (!group_barrier(count, target, n, s_fail)) return false;
        float *t = cur;
        cur = prev;
        prev = t;
    }
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
// CTA.
constexpr int WS_LINE = 32;              // ints of a line (wave_ws_bytes)

// RF: the radius of every grid of the launch (0: per instance)
template <int RF, bool HIST>
__global__ void __launch_bounds__(WAVE_THREADS, 2)
wave_kernel(const GridDev *__restrict__ grids, const Inst *__restrict__ insts, int n_inst, int group, int *ws,
            float *slots, long long slot_floats, int *err, double *partial)
{
    __shared__ float4 xrows[WAVE_THREADS / 32 * XRow<MAX_R>::ROWS * XRow<RF ? RF : MAX_R>::LEN];
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
        const int R = RF ? RF : g.R;
        bool ok;
        if (R == 8)
            ok = RF == 0 || RF == 8 ? run_instance<8, HIST>(g, in, bufA, bufB, xrows, rank, group, count, target, &s_fail, red, gpart, partial) : true;
        else if (R == 4)
            ok = RF == 0 || RF == 4 ? run_instance<4, HIST>(g, in, bufA, bufB, xrows, rank, group, count, target, &s_fail, red, gpart, partial) : true;
        else if (R == 2)
            ok = RF == 0 || RF == 2 ? run_instance<2, HIST>(g, in, bufA, bufB, xrows, rank, group, count, target, &s_fail, red, gpart, partial) : true;
        else
            ok = RF == 0 || RF == 1 ? run_instance<1, HIST>(g, in, bufA, bufB, xrows, rank, group, count, target, &s_fail, red, gpart, partial) : true;
        if (!ok) break;
    }
    if (threadIdx.x == 0 && s_fail) atomicExch(err, EMPSO_TIMEOUT);
}

using WaveFn = void (*)(const GridDev *, const Inst *, int, int, int *, float *, long long, int *, double *);

// (the history only at radius 8: the gradients of the other orders run their
// forward pass on the cluster kernels or per step)
WaveFn wave_fn(int R, bool hist = false)
{
    if (hist) return R == 8 ? wave_kernel<8, true> : nullptr;
    if (R == 8) return wave_kernel<8, false>;
    if (R == 4) return wave_kernel<4, false>;
    if (R == 2) return wave_kernel<2, false>;
    return R == 1 ? wave_kernel<1, false> : wave_kernel<0, false>;
}

}  // namespace

int wave_max_ctas(int R, bool hist)
{
    static std::mutex mu;
    static std::map<std::tuple<int, int, bool>, int> memo;
    int dev = 0, sms = 0, n = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 0;
    std::lock_guard<std::mutex> lock(mu);
    const auto it = memo.find({dev, R, hist});
    if (it != memo.end()) return it->second;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, wave_fn(R, hist), WAVE_THREADS, 0) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return memo[{dev, R, hist}] = std::min(sms * n, WAVE_MAX_CTAS);
}

// Instances in flight and CTAs per instance: the split of the co-resident CTAs
// with the least estimated time, rounds of instances x rows a thread sweeps
// (plus RUN_EXTRA rows' worth for the window it loads first and the step
// barrier), with at most `by_l2` instances in flight
WaveSplit wave_split(const GridDev *const *grids, int n_grids, int R, long long n_inst, long long by_l2,
                     bool hist)
{
    constexpr int RUN_EXTRA = 10;
    WaveSplit best{};
    const int ctas = wave_max_ctas(R, hist);
    const long long most = std::max<long long>(1, std::min<long long>({n_inst, by_l2, (long long)ctas}));
    double cost = 0.0;
    for (long long f = 1; f <= most && ctas > 0; ++f) {
        const int n = (int)(ctas / f);
        long long rows = 0;
        for (int i = 0; i < n_grids; ++i) {
            const GridDev &g = *grids[i];
            const int nth = n * WAVE_THREADS, nseg = std::max(1, std::min(g.NZ, nth / g.NQ));
            rows = std::max<long long>(rows, (long long)((g.NZ + nseg - 1) / nseg) * ((g.NQ * nseg + nth - 1) / nth));
        }
        const double c = (double)((n_inst + f - 1) / f) * (double)(rows + RUN_EXTRA);
        if (best.group == 0 || c < cost) {
            cost = c;
            best.flight = (int)f;
            best.group = n;
        }
    }
    return best;
}

cudaError_t launch_wave(int R, const GridDev *grids_dev, const Inst *insts, int n_inst, const WaveSplit &s,
                        void *ws, float *slots, long long slot_floats, int *err, double *partial, cudaStream_t st,
                        bool hist)
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
    return cudaLaunchKernelEx(&cfg, wave_fn(R, hist), grids_dev, insts, n_inst, s.group, (int *)ws, slots, slot_floats,
                              err, partial);
}

// misfit[p] = sum_s weight_s partial[p][s] in fixed shot order; non-finite
// sums become +inf and are counted in nf[0] (running) and nf[1] (per call).
__global__ void finalize_kernel(const double *partial, const float *weights, int P, int S,
                                double *misfit, unsigned long long *nf)
{
    int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= P) return;
    double s = 0.0;
    for (int k = 0; k < S; ++k) s += (double)weights[k] * partial[(size_t)p * S + k];
    if (!isfinite(s)) {
        s = __longlong_as_double(0x7ff0000000000000LL);
        if (nf) {
            atomicAdd(nf, 1ull);
            atomicAdd(nf + 1, 1ull);
        }
    }
    misfit[p] = s;
}

cudaError_t launch_finalize(const double *partial, const float *weights, int P, int S,
                            double *misfit, unsigned long long *nf, cudaStream_t st)
{
    if (P <= 0) return cudaSuccess;
    finalize_kernel<<<(P + 127) / 128, 128, 0, st>>>(partial, weights, P, S, misfit, nf);
    return cudaGetLastError();
}

}  // namespace empso
