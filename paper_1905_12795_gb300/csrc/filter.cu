// Observed-data preprocessing (section "Testing approach": the recorded data
// are low-pass filtered below the modelling band before the inversion):
// band-limited resampling of traces with the Blackman-windowed sinc
//   h(tau) = 2 fc sinc(2 fc tau) w(tau / W),
//   w(u) = 0.42 + 0.5 cos(pi u) + 0.08 cos(2 pi u) for |u| < 1, else 0,
//   out[s][m][r] = dt_in sum_n in[s][n][r] h(m dt_out - n dt_in),
// records starting at t = 0 and zero outside them.  With dt_out = dt_in it is
// a zero-phase low-pass.
//
// Two kernels (one where few taps are formed: lowpass_narrow_kernel).  lowpass_taps_kernel writes the taps of each tile of LM output
// times, k-major (taps[tile][k][j], k the input sample from the tile's first
// one, j the output time), once for all shots and receivers: their FP64
// arguments run at 1/64 of the FP32 rate, and formed by every (shot, 8 output
// times) block they cost more than the products.  lowpass_kernel is then a
// banded matrix product over all (shot, receiver) columns together: a CTA takes
// LM = 32 NG output times x 32 TC columns, a warp NG groups of 8 times, a lane
// TC columns, in chunks of KC input samples staged by cp.async three deep; the
// taps are read as broadcasts, the products are packed FP32x2 over pairs of
// output times.  Each output sums its input samples in ascending order over the
// window of its group of 8 output times, whatever the tile.  Bound by the FP32
// pipes and the issue slots; 16 shots x 1414 x 461 outputs from 2826-step traces
// with a 0.5 s half-width: 927 -> 421 us (the products 49 of 80 TFLOP/s; the taps 21 us).
#include <algorithm>

#include "internal.cuh"

namespace empso {

namespace {

constexpr int MT = 8;            // output times of a group
constexpr int LTHREADS = 128;    // four warps
template <int NG> constexpr int LMT = LTHREADS / 32 * NG * MT;   // output times of a CTA
constexpr int KC = 16;           // input samples per chunk
constexpr int LSTAGES = 3;

struct LowpassDev {
    int nt_in, nrec, S, nt_out, kpad;       // kpad: taps per output time of a tile (a multiple of KC)
    double dt_in, dt_out, fc, W, invW;
};

// input samples [lo, hi] that outputs m0 .. m0 + count - 1 read
__device__ __forceinline__ void window(const LowpassDev &p, int m0, int count, int &lo, int &hi)
{
    const double t0 = m0 * p.dt_out, t1 = (m0 + count - 1) * p.dt_out;
    lo = max((int)ceil((t0 - p.W) / p.dt_in), 0);
    hi = min((int)floor((t1 + p.W) / p.dt_in), p.nt_in - 1);
}

// The tap of input sample n for the output at time tj.  The argument in FP64: one
// product-sum, two products and two conversions.
__device__ __forceinline__ float tap(const LowpassDev &p, float scale, double tj, int n)
{
    const double tau = fma(-(double)n, p.dt_in, tj);
    const double u = tau * p.invW;
    if ((__double2hiint(u) & 0x7fffffff) >= 0x3ff00000) return 0.f;      // |u| >= 1
    const float uf = (float)u;
    const float w = 0.42f + 0.5f * cospif(uf) + 0.08f * cospif(2.f * uf);
    const float x = (float)(2.0 * p.fc * tau);
    const float sinc = (x == 0.f) ? 1.f : sinpif(x) / (3.14159265358979f * x);
    return scale * sinc * w;
}

// The times of the block's LM outputs are formed once.
template <int NG>
__global__ void __launch_bounds__(256) lowpass_taps_kernel(LowpassDev p, int tile0, float scale, float *taps)
{
    constexpr int LM = LMT<NG>, GROUPS = LM / MT;
    __shared__ int s_lo[GROUPS + 1], s_hi[GROUPS + 1];
    __shared__ double t_out[LM];
    const int m0 = (tile0 + blockIdx.y) * LM;
    if (threadIdx.x <= GROUPS) {            // the tile's window, then its groups'
        const int g = threadIdx.x, a = g == 0 ? m0 : m0 + (g - 1) * MT, n = g == 0 ? LM : MT;
        int lo = 0, hi = -1;
        if (a < p.nt_out) window(p, a, min(n, p.nt_out - a), lo, hi);
        s_lo[g] = lo;
        s_hi[g] = hi;
    }
    for (int j = threadIdx.x; j < LM; j += 256) t_out[j] = (m0 + j) * p.dt_out;
    __syncthreads();
    const int j = threadIdx.x % LM, g = 1 + j / MT;
    const double tj = t_out[j];
    for (int k = blockIdx.x * (256 / LM) + threadIdx.x / LM; k < p.kpad; k += gridDim.x * (256 / LM)) {
        const int n = s_lo[0] + k;
        const float v = m0 + j < p.nt_out && n >= s_lo[g] && n <= s_hi[g] ? tap(p, scale, tj, n) : 0.f;
        taps[((size_t)blockIdx.y * p.kpad + k) * LM + j] = v;
    }
}

// 4 bytes global -> shared, zero where invalid (then nothing is read)
__device__ __forceinline__ void cp4_zfill(float *sdst, const float *gsrc, bool valid)
{
    const unsigned d = (unsigned)__cvta_generic_to_shared(sdst);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;\n" ::"r"(d), "l"(gsrc), "r"(valid ? 4 : 0) : "memory");
}

template <int NG, int TC>
__global__ void __launch_bounds__(LTHREADS)
lowpass_kernel(LowpassDev p, int tile0, const float *__restrict__ in, float *__restrict__ out,
               const float *__restrict__ taps)
{
    constexpr int LM = LMT<NG>, CT = 32 * TC, PER = (CT + LTHREADS - 1) / LTHREADS;    // columns a thread stages
    extern __shared__ __align__(16) float sm[];
    float *xs = sm, *ts = sm + LSTAGES * KC * CT;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int m0 = (tile0 + blockIdx.y) * LM;
    const long long c0 = (long long)blockIdx.x * CT, cols = (long long)p.S * p.nrec;
    int lo, hi;
    window(p, m0, min(LM, p.nt_out - m0), lo, hi);
    const int mw = m0 + warp * NG * MT;
    int k0[NG], k1[NG];                                         // the taps of this warp's groups
#pragma unroll
    for (int g = 0; g < NG; ++g) {
        int glo = 0, ghi = -1;
        if (mw + g * MT < p.nt_out) window(p, mw + g * MT, min(MT, p.nt_out - mw - g * MT), glo, ghi);
        k0[g] = glo - lo;
        k1[g] = ghi - lo + 1;
    }
    const int span = hi >= lo ? hi - lo + 1 : 0, chunks = (span + KC - 1) / KC;
    const float *tp = taps + (size_t)blockIdx.y * p.kpad * LM;
    // the columns this thread stages
    const float *xp[PER];
    bool xok[PER];
#pragma unroll
    for (int i = 0; i < PER; ++i) {
        const int cc = tid + i * LTHREADS;
        const long long c = c0 + cc;
        xok[i] = cc < CT && c < cols;
        const long long s = xok[i] ? c / p.nrec : 0, r = xok[i] ? c % p.nrec : 0;
        xp[i] = in + (s * p.nt_in + lo) * p.nrec + r;
    }
    auto stage = [&](int ch) {
        if (ch < chunks) {
            float *x = xs + (ch % LSTAGES) * KC * CT, *t = ts + (ch % LSTAGES) * KC * LM;
#pragma unroll
            for (int i = 0; i < PER; ++i) {
                if (CT < LTHREADS && tid >= CT) break;
#pragma unroll
                for (int k = 0; k < KC; ++k) {
                    const bool ok = xok[i] && ch * KC + k < span;
                    cp4_zfill(x + k * CT + tid + i * LTHREADS, ok ? xp[i] + (size_t)k * p.nrec : in, ok);
                }
                xp[i] += (size_t)KC * p.nrec;
            }
            // KC x LM taps, 16 bytes at a time (the table is a multiple of KC deep)
#pragma unroll
            for (int q = 0; q < KC * LM / (4 * LTHREADS); ++q) {
                const int o = 4 * (tid + q * LTHREADS);
                const unsigned d = (unsigned)__cvta_generic_to_shared(t + o);
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d), "l"(tp + (size_t)ch * KC * LM + o)
                             : "memory");
            }
        }
        asm volatile("cp.async.commit_group;\n" ::: "memory");
    };
    static_assert(KC * LM % (4 * LTHREADS) == 0, "whole 16-byte copies of the taps per thread");
    float2 acc[NG][MT / 2][TC];
#pragma unroll
    for (int g = 0; g < NG; ++g)
#pragma unroll
        for (int j = 0; j < MT / 2; ++j)
#pragma unroll
            for (int i = 0; i < TC; ++i) acc[g][j][i] = make_float2(0.f, 0.f);
    for (int c = 0; c < LSTAGES - 1; ++c) stage(c);
    for (int ch = 0; ch < chunks; ++ch) {
        asm volatile("cp.async.wait_group %0;\n" ::"n"(LSTAGES - 2) : "memory");
        __syncthreads();
        stage(ch + LSTAGES - 1);            // into the buffer every warp has left
        const float *x = xs + (ch % LSTAGES) * KC * CT + lane, *t = ts + (ch % LSTAGES) * KC * LM + warp * NG * MT;
        // sample k of the chunk, for the groups whose window holds it
        auto term = [&](int k, auto on) {
            float v[TC];
#pragma unroll
            for (int i = 0; i < TC; ++i) v[i] = x[k * CT + 32 * i];
#pragma unroll
            for (int g = 0; g < NG; ++g) {
                if (!on(g)) continue;
                const float4 a = *reinterpret_cast<const float4 *>(t + k * LM + g * MT);
                const float4 b = *reinterpret_cast<const float4 *>(t + k * LM + g * MT + 4);
#pragma unroll
                for (int i = 0; i < TC; ++i) {
                    const float2 vv = make_float2(v[i], v[i]);
                    acc[g][0][i] = __ffma2_rn(make_float2(a.x, a.y), vv, acc[g][0][i]);
                    acc[g][1][i] = __ffma2_rn(make_float2(a.z, a.w), vv, acc[g][1][i]);
                    acc[g][2][i] = __ffma2_rn(make_float2(b.x, b.y), vv, acc[g][2][i]);
                    acc[g][3][i] = __ffma2_rn(make_float2(b.z, b.w), vv, acc[g][3][i]);
                }
            }
        };
        const int base = ch * KC;
        bool whole = true;
#pragma unroll
        for (int g = 0; g < NG; ++g) whole = whole && k0[g] <= base && k1[g] >= base + KC;
        if (whole) {
#pragma unroll
            for (int k = 0; k < KC; ++k) term(k, [](int) { return true; });
        } else {
            for (int k = 0; k < KC; ++k)
                term(k, [&](int g) { return k0[g] <= base + k && base + k < k1[g]; });
        }
    }
    asm volatile("cp.async.wait_group 0;\n" ::: "memory");
#pragma unroll
    for (int i = 0; i < TC; ++i) {
        const long long c = c0 + lane + 32 * i;
        if (c >= cols) continue;
        const long long s = c / p.nrec, r = c % p.nrec;
        float *o = out + (s * p.nt_out + mw) * p.nrec + r;
#pragma unroll
        for (int j = 0; j < NG * MT; ++j) {
            const float2 v = acc[j / MT][j % MT / 2][i];
            if (mw + j < p.nt_out) o[(size_t)j * p.nrec] = (j & 1) ? v.y : v.x;
        }
    }
}

// Short windows: one launch, a CTA forms the taps of 8 output times in shared memory
// and takes them over NARROW_COLS columns, one per thread.  The table's second launch
// costs more than forming the taps again in every CTA while few are formed, up to about
// a million: 16 shots x 150 x 461 outputs, 56 input samples each, 28 us against 40 with
// the table; 4 x 250 x 162 outputs of 200 samples (150,000 taps) 28 against 36; 16 x 400
// x 461 of 160 (1.9 million) 60 against 54.  Each output is the sum that lowpass_kernel forms, in its order.
constexpr int NARROW_SPAN = 256, NARROW_COLS = 256;
constexpr long long NARROW_TAPS = 1 << 20;
__global__ void __launch_bounds__(NARROW_COLS)
lowpass_narrow_kernel(LowpassDev p, float scale, const float *__restrict__ in, float *__restrict__ out)
{
    __shared__ __align__(16) float taps[NARROW_SPAN * MT];
    const int m0 = blockIdx.y * MT, count = min(MT, p.nt_out - m0);
    int lo, hi;
    window(p, m0, count, lo, hi);
    const int span = hi >= lo ? min(hi - lo + 1, NARROW_SPAN) : 0;
    for (int e = threadIdx.x; e < span * MT; e += NARROW_COLS) {
        const int j = e % MT;
        taps[e] = j < count ? tap(p, scale, (m0 + j) * p.dt_out, lo + e / MT) : 0.f;
    }
    __syncthreads();
    const long long c = (long long)blockIdx.x * NARROW_COLS + threadIdx.x;
    if (c >= (long long)p.S * p.nrec) return;
    const long long s = c / p.nrec, r = c % p.nrec;
    const float *x = in + (s * p.nt_in + lo) * p.nrec + r;
    float2 acc[MT / 2];
#pragma unroll
    for (int j = 0; j < MT / 2; ++j) acc[j] = make_float2(0.f, 0.f);
#pragma unroll 4
    for (int k = 0; k < span; ++k) {
        const float v = __ldg(x + (size_t)k * p.nrec);
        const float2 vv = make_float2(v, v);
#pragma unroll
        for (int j = 0; j < MT / 2; ++j)
            acc[j] = __ffma2_rn(*reinterpret_cast<const float2 *>(taps + k * MT + 2 * j), vv, acc[j]);
    }
    float *o = out + (s * p.nt_out + m0) * p.nrec + r;
#pragma unroll
    for (int j = 0; j < MT; ++j)
        if (j < count) o[(size_t)j * p.nrec] = (j & 1) ? acc[j / 2].y : acc[j / 2].x;
}

// input samples that 8 output times read, at most
long long lowpass_span(double dt_in, double dt_out, double W)
{
    return (long long)std::ceil(((MT - 1) * dt_out + 2.0 * W) / dt_in) + 2;
}

bool lowpass_narrow(long long cols, int nt_in, int nt_out, double dt_in, double dt_out, double W)
{
    const long long span = std::min<long long>(lowpass_span(dt_in, dt_out, W), nt_in);
    return span <= NARROW_SPAN && (cols + NARROW_COLS - 1) / NARROW_COLS * nt_out * span <= NARROW_TAPS;
}

int lowpass_kpad(int LM, double dt_in, double dt_out, double W)
{
    const long long span = (long long)std::ceil(((LM - 1) * dt_out + 2.0 * W) / dt_in) + 2;
    return (int)((span + KC - 1) / KC * KC);
}

// The widest tile that still gives every SM four CTAs: 16 output times x 4
// columns a thread (the fewest shared-memory reads and copies per product that
// leave four CTAs per SM their registers), then 8 x 4, 8 x 2, 8 x 1.
struct LowpassShape {
    int NG, TC;
};
LowpassShape lowpass_shape(long long cols, int nt_out, int sms)
{
    const LowpassShape shapes[] = {{2, 4}, {1, 4}, {1, 2}, {1, 1}};
    for (const LowpassShape &s : shapes) {
        const int LM = LTHREADS / 32 * s.NG * MT;
        if ((cols + 32 * s.TC - 1) / (32 * s.TC) * ((nt_out + LM - 1) / LM) >= 4LL * sms) return s;
    }
    return {1, 1};
}

template <int NG, int TC>
cudaError_t lowpass_pass(const LowpassDev &p, int t0, int n, const float *in, float *out, float *ws, cudaStream_t st)
{
    constexpr int LM = LMT<NG>;
    constexpr size_t smem = sizeof(float) * LSTAGES * KC * (32 * TC + LM);
    static_assert(smem <= 48 << 10, "no opt-in");
    const int blocks = (p.kpad + 256 / LM - 1) / (256 / LM);
    lowpass_taps_kernel<NG><<<dim3((blocks + 3) / 4, n), 256, 0, st>>>(p, t0, (float)(p.dt_in * 2.0 * p.fc), ws);
    const long long cols = (long long)p.S * p.nrec;
    lowpass_kernel<NG, TC><<<dim3((unsigned)((cols + 32 * TC - 1) / (32 * TC)), n), LTHREADS, smem, st>>>(p, t0, in, out, ws);
    return cudaGetLastError();
}

}  // namespace

// largest input window of 8 output times; a window whose taps for 8 output times
// exceed `limit` bytes (the shared memory of a CTA) is not supported
bool lowpass_supported(double dt_in, double dt_out, double W, size_t limit)
{
    return sizeof(float) * MT * (size_t)lowpass_span(dt_in, dt_out, W) <= limit;
}

// workspace floats of the taps: all tiles', or as many as MOST holds (then the
// call takes several passes), at least one tile's; 0: the call needs no table
size_t lowpass_ws_floats(int S, int nt_in, int nrec, int nt_out, double dt_in, double dt_out, double W, int sms)
{
    constexpr size_t MOST = 16u << 20;      // 64 MB
    if (lowpass_narrow((long long)S * nrec, nt_in, nt_out, dt_in, dt_out, W)) return 0;
    const int LM = LTHREADS / 32 * MT * lowpass_shape((long long)S * nrec, nt_out, sms).NG;
    const size_t tile = (size_t)lowpass_kpad(LM, dt_in, dt_out, W) * LM, tiles = (nt_out + LM - 1) / LM;
    return tile * std::max<size_t>(1, std::min(tiles, MOST / tile));
}

cudaError_t launch_lowpass(const float *in, int S, int nt_in, int nrec, double dt_in, float *out,
                           int nt_out, double dt_out, double fc, double W, float *ws, size_t ws_floats, int sms,
                           cudaStream_t st)
{
    const LowpassShape shape = lowpass_shape((long long)S * nrec, nt_out, sms);
    const int LM = LTHREADS / 32 * MT * shape.NG, tiles = (nt_out + LM - 1) / LM;
    LowpassDev p{nt_in, nrec, S, nt_out, lowpass_kpad(LM, dt_in, dt_out, W), dt_in, dt_out, fc, W, 1.0 / W};
    const long long cols = (long long)S * nrec;
    if (lowpass_narrow(cols, nt_in, nt_out, dt_in, dt_out, W)) {
        const dim3 grid((unsigned)((cols + NARROW_COLS - 1) / NARROW_COLS), (nt_out + MT - 1) / MT);
        lowpass_narrow_kernel<<<grid, NARROW_COLS, 0, st>>>(p, (float)(dt_in * 2.0 * fc), in, out);
        return cudaGetLastError();
    }
    const int pass = (int)std::min<size_t>({(size_t)tiles, ws_floats / ((size_t)p.kpad * LM), (size_t)65535});
    for (int t0 = 0; t0 < tiles; t0 += pass) {
        const int n = std::min(pass, tiles - t0);
        const cudaError_t e = shape.NG == 2   ? lowpass_pass<2, 4>(p, t0, n, in, out, ws, st)
                              : shape.TC == 4 ? lowpass_pass<1, 4>(p, t0, n, in, out, ws, st)
                              : shape.TC == 2 ? lowpass_pass<1, 2>(p, t0, n, in, out, ws, st)
                                              : lowpass_pass<1, 1>(p, t0, n, in, out, ws, st);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace empso
