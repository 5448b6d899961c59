// Surrogate network that pre-screens EMPSO particles (the paper has none; it
// serves the pre-screening pattern the library adds): a K -> H -> H -> 1
// ReLU perceptron predicting the standardised log-misfit of a particle from
// its control nodes scaled to [-1, 1].  Dense layers run on the tensor cores
// (BF16 operands, FP32 accumulation), master weights and Adam moments are
// FP32, and the training set is a device-side replay buffer filled with the
// (particle, misfit) pairs the fitness evaluation produces.
#include <cooperative_groups.h>
#include <cuda_bf16.h>

#include <utility>

#include "internal.cuh"

namespace empso {

namespace {

// ---------------------------------------------------------------------------
// C[M][N] = sum_k A(m, k) B(k, n) (+ bias[n], ReLU) with BF16 operands and
// FP32 accumulation on mma.sync m16n8k16.  A(m, k) = A[m lda + k] (a_mk) or
// A[k lda + m]; B(k, n) = B[n ldb + k] (b_nk) or B[k ldb + n].  Tiles of
// 64 x 64 per 128-thread block, 32-deep k-steps staged in shared memory
// (zero-filled past M, N, K).  Outputs: FP32 Cf and/or BF16 Cb.
// ---------------------------------------------------------------------------
constexpr int GBM = 64, GBN = 64, GBK = 32, GPAD = 8;

// One product and what becomes of it: v = C + bias[n], ReLU, or zero where the
// mask (BF16 [M][ldm]) is not positive; FP32 Cf and/or BF16 Cb.
struct Gemm {
    int M, N, K;
    const __nv_bfloat16 *A;
    int lda, a_mk;
    const __nv_bfloat16 *B;
    int ldb, b_nk;
    const float *bias;
    int relu;
    const __nv_bfloat16 *mask;
    int ldm;
    float *Cf;
    int ldc;
    __nv_bfloat16 *Cb;
    int ldcb;
};

__device__ __forceinline__ void mma_bf16(float c[4], const unsigned a[4], const unsigned b[2])
{
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, "
        "{%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

__global__ void __launch_bounds__(128) gemm_bf16_kernel(const Gemm g)
{
    const int M = g.M, N = g.N, K = g.K, lda = g.lda, a_mk = g.a_mk, ldb = g.ldb, b_nk = g.b_nk;
    const __nv_bfloat16 *__restrict__ A = g.A, *__restrict__ B = g.B;
    __shared__ __align__(16) __nv_bfloat16 As[GBM][GBK + GPAD];   // (m, k)
    __shared__ __align__(16) __nv_bfloat16 Bs[GBN][GBK + GPAD];   // (n, k)
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int lg = lane >> 2, t = lane & 3;
    const int m0 = blockIdx.y * GBM, n0 = blockIdx.x * GBN;
    const int wm = (warp >> 1) * 32, wn = (warp & 1) * 32;
    float acc[2][4][4];
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int e = 0; e < 4; ++e) acc[i][j][e] = 0.f;
    const __nv_bfloat16 zero = __float2bfloat16(0.f);
    for (int k0 = 0; k0 < K; k0 += GBK) {
        for (int e = tid; e < GBM * GBK; e += 128) {
            int mm, kk;
            if (a_mk) { mm = e / GBK; kk = e % GBK; } else { kk = e / GBM; mm = e % GBM; }
            const int m = m0 + mm, k = k0 + kk;
            __nv_bfloat16 v = zero;
            if (m < M && k < K) v = a_mk ? A[(size_t)m * lda + k] : A[(size_t)k * lda + m];
            As[mm][kk] = v;
        }
        for (int e = tid; e < GBN * GBK; e += 128) {
            int nn, kk;
            if (b_nk) { nn = e / GBK; kk = e % GBK; } else { kk = e / GBN; nn = e % GBN; }
            const int n = n0 + nn, k = k0 + kk;
            __nv_bfloat16 v = zero;
            if (n < N && k < K) v = b_nk ? B[(size_t)n * ldb + k] : B[(size_t)k * ldb + n];
            Bs[nn][kk] = v;
        }
        __syncthreads();
#pragma unroll
        for (int ks = 0; ks < GBK; ks += 16) {
            unsigned af[2][4], bf[4][2];
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                const int r = wm + 16 * i + lg;
                af[i][0] = *reinterpret_cast<const unsigned *>(&As[r][ks + 2 * t]);
                af[i][1] = *reinterpret_cast<const unsigned *>(&As[r + 8][ks + 2 * t]);
                af[i][2] = *reinterpret_cast<const unsigned *>(&As[r][ks + 2 * t + 8]);
                af[i][3] = *reinterpret_cast<const unsigned *>(&As[r + 8][ks + 2 * t + 8]);
            }
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int c = wn + 8 * j + lg;
                bf[j][0] = *reinterpret_cast<const unsigned *>(&Bs[c][ks + 2 * t]);
                bf[j][1] = *reinterpret_cast<const unsigned *>(&Bs[c][ks + 2 * t + 8]);
            }
#pragma unroll
            for (int i = 0; i < 2; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) mma_bf16(acc[i][j], af[i], bf[j]);
        }
        __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int m = m0 + wm + 16 * i + lg + (e >= 2 ? 8 : 0);
                const int n = n0 + wn + 8 * j + 2 * t + (e & 1);
                if (m >= M || n >= N) continue;
                float v = acc[i][j][e];
                if (g.bias) v += g.bias[n];
                if (g.relu) v = fmaxf(v, 0.f);
                if (g.mask && !(__bfloat162float(g.mask[(size_t)m * g.ldm + n]) > 0.f)) v = 0.f;
                if (g.Cf) g.Cf[(size_t)m * g.ldc + n] = v;
                if (g.Cb) g.Cb[(size_t)m * g.ldcb + n] = __float2bfloat16(v);
            }
}

// ---------------------------------------------------------------------------
// The same product on the 5th-generation tensor cores: tcgen05.mma with BF16
// operands from shared memory and the FP32 accumulator in tensor memory.
// One CTA (8 warps) computes a 128 x NT tile (NT = 64, or N rounded up to 16
// when N < 64) over k-chunks of up to TKC = 256: the whole depth of a forward or
// data-gradient product, so that all its loads are in flight together; deeper
// products (the weight gradients, whose depth is the batch) are
// double-buffered.  Staging writes the K-major canonical layout without swizzle
// (8-row x 16-byte core matrices; the two 8-element halves of a 16-deep k-slice
// 128 bytes apart, successive 8-row groups 256 bytes apart): rows stored
// k-fastest are copied 16 bytes at a time, operands stored m/n-fastest are
// transposed in registers 8 x 8 elements at a time.  One thread issues a
// 128 x NT x 16 MMA per k-slice and commits a chunk's to the buffer's mbarrier;
// after the last chunk every warp reads its 32 accumulator rows of every other
// 16 columns with tcgen05.ld for the epilogue.  Bound by latency (launch, one
// round of global loads, the epilogue), not by the tensor core: with 64-deep
// chunks and 128 threads each chunk waited for its own loads, 25 us for 1024 x
// 256 x 256 and 45 us for 256 x 256 x 1024 (ncu); now 17 and 26 us.
// ---------------------------------------------------------------------------
constexpr int TM = 128, TKC = 256, TNT = 64, TC_THREADS = 256;
constexpr int TC_SMEM = 2 * (TKC / 16) * (TM + TNT) * 32;   // two k-chunk buffers
__host__ __device__ inline int tc_tile_n(int N) { return N >= TNT ? TNT : (N + 15) / 16 * 16; }

__device__ __forceinline__ unsigned smem_u32(const void *p) { return (unsigned)__cvta_generic_to_shared(p); }

// no-swizzle K-major descriptor: start >> 4, LBO (k-direction core stride) >> 4,
// SBO (m/n-direction core stride) >> 4, descriptor version 1
__device__ __forceinline__ unsigned long long umma_desc(const void *p, unsigned lbo, unsigned sbo)
{
    unsigned long long d = 0;
    d |= (unsigned long long)((smem_u32(p) >> 4) & 0x3FFF);
    d |= (unsigned long long)((lbo >> 4) & 0x3FFF) << 16;
    d |= (unsigned long long)((sbo >> 4) & 0x3FFF) << 32;
    d |= 1ull << 46;
    return d;
}

// kind::f16 instruction descriptor: D FP32, A and B BF16, both K-major,
// N >> 3 at bit 17, M >> 4 at bit 24
__device__ __forceinline__ unsigned umma_idesc(int M, int N)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | ((unsigned)(N >> 3) << 17) | ((unsigned)(M >> 4) << 24);
}

// byte offset of element (row r, k) inside a 16-deep k-slice of a K-major tile
__device__ __forceinline__ int canon_off(int r, int k)
{
    return (r >> 3) * 256 + (k >> 3) * 128 + (r & 7) * 16 + (k & 7) * 2;
}

__device__ __forceinline__ bool mbar_try(unsigned addr, unsigned parity)
{
    unsigned ok;
    asm volatile("{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
                 " selp.u32 %0, 1, 0, p;\n}\n"
                 : "=r"(ok)
                 : "r"(addr), "r"(parity)
                 : "memory");
    return ok != 0;
}

// wait (at most WAIT_LIMIT_NS) for the phase of `parity` of an mbarrier
__device__ __forceinline__ bool mbar_wait_tc(unsigned addr, unsigned parity)
{
    if (mbar_try(addr, parity)) return true;
    const unsigned long long t0 = global_ns();
    for (;;) {
        if (mbar_try(addr, parity)) return true;
        if (global_ns() - t0 > WAIT_LIMIT_NS) return false;
    }
}

// Stage rows r0 .. r0 + R - 1 (of M) x k0 .. k0 + kc - 1 (of K; kc a multiple
// of 16) of an operand into the canonical layout at dst (kc / 16 slices of R x
// 16 elements).  kmajor: element (r, k) at src[r ld + k]; otherwise at
// src[k ld + r].  vec: ld % 8 == 0 and src 16-byte aligned (16-byte accesses
// allowed).
__device__ __forceinline__ void stage_operand(unsigned char *dst, const __nv_bfloat16 *__restrict__ src,
                                              int ld, int kmajor, bool vec, int r0, int R, int M,
                                              int k0, int kc, int K)
{
    const int tid = threadIdx.x;
    const __nv_bfloat16 zero = __float2bfloat16(0.f);
    if (vec && kmajor) {
        // one 16-byte vector = 8 consecutive k of one row; a warp takes 8 rows
        // (one core matrix, every bank once) by 2 or 4 vectors (whole sectors)
        const int nkv = kc / 8, kg = nkv % 4 == 0 ? 4 : 2;
        const int per = 8 * kg, blocks_k = nkv / kg;
#pragma unroll 8
        for (int v = tid; v < R * nkv; v += TC_THREADS) {
            const int in = v % per, blk = v / per;
            const int r = (blk / blocks_k) * 8 + (in & 7), kv = ((blk % blocks_k) * kg + (in >> 3)) * 8;
            const int row = r0 + r, k = k0 + kv;
            uint4 val = make_uint4(0u, 0u, 0u, 0u);
            if (row < M) {
                const __nv_bfloat16 *p = src + (size_t)row * ld + k;
                if (k + 8 <= K) {
                    val = *reinterpret_cast<const uint4 *>(p);
                } else if (k < K) {
                    __nv_bfloat16 t[8];
                    for (int e = 0; e < 8; ++e) t[e] = (k + e < K) ? p[e] : zero;
                    val = *reinterpret_cast<const uint4 *>(t);
                }
            }
            *reinterpret_cast<uint4 *>(dst + (kv >> 4) * (R * 32) + canon_off(r, kv & 15)) = val;
        }
    } else if (vec && (M & 7) == 0) {
        // 8 (rows) x 8 (k) blocks: eight 16-byte loads along the rows, a
        // register transpose, eight 16-byte stores along k
        for (int b = tid; b < (R / 8) * (kc / 8); b += TC_THREADS) {
            const int rb = (b % (R / 8)) * 8, kb = (b / (R / 8)) * 8;
            const int row = r0 + rb;
            uint4 in[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const int k = k0 + kb + i;
                in[i] = (row < M && k < K)
                            ? *reinterpret_cast<const uint4 *>(src + (size_t)k * ld + row)
                            : make_uint4(0u, 0u, 0u, 0u);
            }
            // word j of in[i] holds rows (2j, 2j+1) at k = i; word i of out[m]
            // must hold k = (2i, 2i+1) at row m
            unsigned o[8][4];
            const unsigned *w = reinterpret_cast<const unsigned *>(in);
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const unsigned a = w[(2 * i) * 4 + j], c = w[(2 * i + 1) * 4 + j];
                    o[2 * j][i] = __byte_perm(a, c, 0x5410);
                    o[2 * j + 1][i] = __byte_perm(a, c, 0x7632);
                }
#pragma unroll
            for (int m = 0; m < 8; ++m)
                *reinterpret_cast<uint4 *>(dst + (kb >> 4) * (R * 32) + canon_off(rb + m, kb & 15)) =
                    make_uint4(o[m][0], o[m][1], o[m][2], o[m][3]);
        }
    } else {
        for (int e = tid; e < R * kc; e += TC_THREADS) {
            int r, kk;
            if (kmajor) { r = e / kc; kk = e % kc; } else { kk = e / R; r = e % R; }
            const int row = r0 + r, k = k0 + kk;
            __nv_bfloat16 v = zero;
            if (row < M && k < K) v = kmajor ? src[(size_t)row * ld + k] : src[(size_t)k * ld + row];
            *reinterpret_cast<__nv_bfloat16 *>(dst + (kk >> 4) * (R * 32) + canon_off(r, kk & 15)) = v;
        }
    }
}

// tile (bx, by) of one product; a CTA's whole work
__device__ __forceinline__ void gemm_tc_tile(const Gemm &g, int bx, int by, int *err)
{
    extern __shared__ __align__(1024) unsigned char tsm[];
    __shared__ __align__(8) unsigned long long mbar[2];
    __shared__ unsigned tmem_base;
    __shared__ int s_fail;
    const int M = g.M, N = g.N, K = g.K;
    const int NT = tc_tile_n(N);
    const int stage_bytes = (TKC / 16) * (TM + NT) * 32;
    const int tid = threadIdx.x, warp = tid >> 5;
    const int m0 = by * TM, n0 = bx * NT;
    const bool a_vec = g.lda % 8 == 0 && ((size_t)g.A & 15) == 0, b_vec = g.ldb % 8 == 0 && ((size_t)g.B & 15) == 0;
    const unsigned ncols = NT <= 32 ? 32u : 64u;        // tensor-memory columns (power of 2)
    if (tid == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(smem_u32(&mbar[0])) : "memory");
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(smem_u32(&mbar[1])) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
        s_fail = 0;
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(
                         smem_u32(&tmem_base)),
                     "r"(ncols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    const unsigned tmem = tmem_base;
    const unsigned idesc = umma_idesc(TM, NT);
    const int nchunks = (K + TKC - 1) / TKC;
    for (int c = 0; c < nchunks; ++c) {
        const int buf = c & 1;
        unsigned char *As = tsm + buf * stage_bytes;
        unsigned char *Bs = As + (TKC / 16) * TM * 32;
        const int kc = min(TKC, (K - c * TKC + 15) / 16 * 16);
        // the MMAs that read this buffer two chunks ago are done before it is restaged
        if (c >= 2 && !mbar_wait_tc(smem_u32(&mbar[buf]), ((c - 2) >> 1) & 1)) s_fail = 1;
        stage_operand(As, g.A, g.lda, g.a_mk, a_vec, m0, TM, M, c * TKC, kc, K);
        stage_operand(Bs, g.B, g.ldb, g.b_nk, b_vec, n0, NT, N, c * TKC, kc, K);
        // thread-written shared memory -> visible to the tensor core (async proxy)
        asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
        __syncthreads();
        if (tid == 0) {
            asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
            for (int s = 0; s < kc / 16; ++s) {
                const unsigned long long ad = umma_desc(As + s * (TM * 32), 128, 256);
                const unsigned long long bd = umma_desc(Bs + s * (NT * 32), 128, 256);
                const unsigned acc = (c > 0 || s > 0) ? 1u : 0u;
                asm volatile("{\n .reg .pred p;\n setp.ne.u32 p, %4, 0;\n"
                             " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem),
                             "l"(ad), "l"(bd), "r"(idesc), "r"(acc)
                             : "memory");
            }
            asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(
                             smem_u32(&mbar[buf]))
                         : "memory");
        }
    }
    // the last commit covers every MMA issued before it
    {
        const int c = nchunks - 1;
        if (!mbar_wait_tc(smem_u32(&mbar[c & 1]), (c >> 1) & 1)) s_fail = 1;
    }
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    __syncthreads();
    // epilogue: warp w reads accumulator rows 32 (w mod 4) .. + 31 (TMEM lanes),
    // warps 0-3 the even blocks of 16 columns, warps 4-7 the odd ones
    const int row = m0 + 32 * (warp & 3) + (tid & 31);
    const bool fail = s_fail != 0;
    for (int c0 = 16 * (warp >> 2); c0 < NT; c0 += 32) {
        unsigned r[16];
        const unsigned taddr = tmem + ((unsigned)(32 * (warp & 3)) << 16) + (unsigned)c0;
        asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n"
                     : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]),
                       "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]),
                       "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
                     : "r"(taddr)
                     : "memory");
        asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
        if (row >= M || fail) continue;
        const int nb = n0 + c0;
        float v[16];
#pragma unroll
        for (int j = 0; j < 16; ++j) {
            float t = __uint_as_float(r[j]);
            if (g.bias && nb + j < N) t += g.bias[nb + j];
            if (g.relu) t = fmaxf(t, 0.f);
            if (g.mask && nb + j < N && !(__bfloat162float(g.mask[(size_t)row * g.ldm + nb + j]) > 0.f)) t = 0.f;
            v[j] = t;
        }
        if (nb + 16 <= N) {
            if (g.Cf) {
                float *o = g.Cf + (size_t)row * g.ldc + nb;
                if ((g.ldc & 3) == 0 && ((size_t)g.Cf & 15) == 0) {
#pragma unroll
                    for (int q = 0; q < 4; ++q)
                        reinterpret_cast<float4 *>(o)[q] = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
                } else {
                    for (int j = 0; j < 16; ++j) o[j] = v[j];
                }
            }
            if (g.Cb) {
                __nv_bfloat16 *o = g.Cb + (size_t)row * g.ldcb + nb;
                if ((g.ldcb & 7) == 0 && ((size_t)g.Cb & 15) == 0) {
                    __nv_bfloat162 h[8];
#pragma unroll
                    for (int q = 0; q < 8; ++q) h[q] = __floats2bfloat162_rn(v[2 * q], v[2 * q + 1]);
                    reinterpret_cast<uint4 *>(o)[0] = *reinterpret_cast<uint4 *>(&h[0]);
                    reinterpret_cast<uint4 *>(o)[1] = *reinterpret_cast<uint4 *>(&h[4]);
                } else {
                    for (int j = 0; j < 16; ++j) o[j] = __float2bfloat16(v[j]);
                }
            }
        } else {
            for (int j = 0; j < 16; ++j) {
                const int n = nb + j;
                if (n >= N) break;
                if (g.Cf) g.Cf[(size_t)row * g.ldc + n] = v[j];
                if (g.Cb) g.Cb[(size_t)row * g.ldcb + n] = __float2bfloat16(v[j]);
            }
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(ncols) : "memory");
    if (tid == 0 && s_fail) atomicExch(err, EMPSO_TIMEOUT);
}

// Column sums g[h] = sum_b v[b][h] over the batch, v = X, or relu(X) times
// wrow[b]: 32 columns per CTA; the partial sum (x, y) takes rows y, y + 32, ...
// of column x, then the 32 partial sums of a column are added pairwise in a
// fixed tree (the same order on every call and for any block size).
constexpr int CS_T = 32;
struct ColSum {
    const float *X, *wrow;
    int n, H;
    float *g;
};
__device__ __forceinline__ void colsum_cols(const ColSum &c, int bx)
{
    __shared__ float red[CS_T][CS_T + 1];
    const int tx = threadIdx.x % CS_T, h = bx * CS_T + tx, step = blockDim.x / CS_T;
    for (int ty = threadIdx.x / CS_T; ty < CS_T; ty += step) {
        float s = 0.f;
        if (h < c.H)
#pragma unroll 8
            for (int b = ty; b < c.n; b += CS_T) {
                const float v = c.X[(size_t)b * c.H + h];
                s = c.wrow ? fmaf(fmaxf(v, 0.f), c.wrow[b], s) : s + v;
            }
        red[ty][tx] = s;
    }
    __syncthreads();
    for (int st = CS_T / 2; st > 0; st >>= 1) {
        for (int ty = threadIdx.x / CS_T; ty < st; ty += step) red[ty][tx] += red[ty + st][tx];
        __syncthreads();
    }
    if (threadIdx.x < CS_T && h < c.H) c.g[h] = red[0][tx];
}

// out = sum_i v[i]: one CTA, 1024 strided partial sums, then a fixed tree
__device__ __forceinline__ void sum_all(const float *__restrict__ v, int n, float *out)
{
    __shared__ float red[1024];
    for (int t = threadIdx.x; t < 1024; t += blockDim.x) {
        float s = 0.f;
        for (int i = t; i < n; i += 1024) s += v[i];
        red[t] = s;
    }
    __syncthreads();
    for (int st = 512; st > 0; st >>= 1) {
        for (int t = threadIdx.x; t < st; t += blockDim.x) red[t] += red[t + st];
        __syncthreads();
    }
    if (threadIdx.x == 0) *out = red[0];
}

// the loss 1/(2n) sum (y - t)^2 (one CTA of 256 threads or more, fixed order)
__device__ __forceinline__ void loss_sum(const float *__restrict__ y, const float *__restrict__ t, int n, float *loss)
{
    __shared__ double red[8];
    if (threadIdx.x < 256) {
        double s = 0.0;
        for (int b = threadIdx.x; b < n; b += 256) {
            const float r = y[b] - t[b];
            s += (double)r * r;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
        if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double v = 0.0;
        for (int w = 0; w < 8; ++w) v += red[w];
        if (loss) *loss = (float)(0.5 * v / n);
    }
}

// Independent parts of the backward pass in one launch: up to two products,
// up to two column sums, the sum of dy and the loss (the small parts would
// each wait for a launch and leave the GPU idle: with these, the fused minibatch
// and the fused head, a training step of 1024 pairs, K = 32, H = 256, takes 7
// launches instead of 17, and six steps and a prediction 584 us instead of 1169).
struct Jobs {
    Gemm g[2];
    ColSum c[2];
    int n_gemm = 0, n_col = 0, sums = 0;
    const float *dy = nullptr, *y = nullptr, *t = nullptr;   // sums: sum of dy into gb3, the loss
    int n = 0;
    float *gb3 = nullptr, *loss = nullptr;
};

__host__ __device__ inline int tc_tiles(const Gemm &g)
{
    const int NT = tc_tile_n(g.N);
    return (g.N + NT - 1) / NT * ((g.M + TM - 1) / TM);
}

// part b of the jobs' vector work: the column sums' CTAs, then dy's sum and the loss
__device__ __forceinline__ void vector_job(const Jobs &j, int b)
{
    for (int i = 0; i < j.n_col; ++i) {
        const int n = (j.c[i].H + CS_T - 1) / CS_T;
        if (b < n) return colsum_cols(j.c[i], b);
        b -= n;
    }
    if (b == 0) sum_all(j.dy, j.n, j.gb3);
    else loss_sum(j.y, j.t, j.n, j.loss);
}

__host__ inline int vector_blocks(const Jobs &j)
{
    int n = j.sums ? 2 : 0;
    for (int i = 0; i < j.n_col; ++i) n += (j.c[i].H + CS_T - 1) / CS_T;
    return n;
}

__global__ void __launch_bounds__(TC_THREADS) jobs_tc_kernel(const Jobs j, int *err)
{
    int b = blockIdx.x;
    for (int i = 0; i < j.n_gemm; ++i) {
        const int n = tc_tiles(j.g[i]);
        if (b < n) {
            const int nx = (j.g[i].N + tc_tile_n(j.g[i].N) - 1) / tc_tile_n(j.g[i].N);
            return gemm_tc_tile(j.g[i], b % nx, b / nx, err);
        }
        b -= n;
    }
    vector_job(j, b);
}

// (1024 threads: a column sum's threads wait for loads; a gradient over 2000 rows on
// mma.sync, K = 32, H = 256, took 468 us with 256 of them, 424 with 1024)
constexpr int VEC_THREADS = 1024;
__global__ void __launch_bounds__(VEC_THREADS) jobs_vector_kernel(const Jobs j) { vector_job(j, blockIdx.x); }

// the jobs on the context's backend: one launch on tcgen05, else one per product
cudaError_t run_jobs(const SurDev &s, const Jobs &j, cudaStream_t st)
{
    const int vb = vector_blocks(j);
    if (s.tc && s.err) {
        int n = vb;
        for (int i = 0; i < j.n_gemm; ++i) n += tc_tiles(j.g[i]);
        if (n > 0) jobs_tc_kernel<<<n, TC_THREADS, j.n_gemm ? TC_SMEM : 0, st>>>(j, s.err);
        return cudaGetLastError();
    }
    for (int i = 0; i < j.n_gemm; ++i) {
        const Gemm &g = j.g[i];
        gemm_bf16_kernel<<<dim3((g.N + GBN - 1) / GBN, (g.M + GBM - 1) / GBM), 128, 0, st>>>(g);
    }
    if (vb) jobs_vector_kernel<<<vb, VEC_THREADS, 0, st>>>(j);
    return cudaGetLastError();
}

cudaError_t run_gemm(const SurDev &s, const Gemm &g, cudaStream_t st)
{
    Jobs j;
    j.g[0] = g;
    j.n_gemm = 1;
    return run_jobs(s, j, st);
}

// ---------------------------------------------------------------------------
// elementwise and reduction kernels
// ---------------------------------------------------------------------------

// x_n = 2 (x - xmin) / (xmax - xmin) - 1 as BF16
__device__ __forceinline__ __nv_bfloat16 normalized(float x, int k, const double *__restrict__ xmin,
                                                    const double *__restrict__ xmax)
{
    const float lo = (float)xmin[k], hi = (float)xmax[k];
    return __float2bfloat16(2.f * (x - lo) / (hi - lo) - 1.f);
}

__global__ void normalize_kernel(const float *__restrict__ x, int n, int K, const double *__restrict__ xmin,
                                 const double *__restrict__ xmax, __nv_bfloat16 *out)
{
    const long long tot = (long long)n * K;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < tot;
         e += (long long)gridDim.x * blockDim.x)
        out[e] = normalized(x[e], (int)(e % K), xmin, xmax);
}

// The head, one warp per row b (fixed order): y = sum_h relu(Z2[b][h]) w3[h] +
// b3.  Predicting (stats given): out[b] = y sigma + mu.  Training (t given):
// also dy = (y - t) / n and, while the row is at hand, the gradient of the
// hidden layer dZ2 = dy w3 [Z2 > 0] (FP32 and BF16 copies).
__global__ void head_kernel(const float *__restrict__ Z2, int n, int H, const float *__restrict__ w3,
                            const float *__restrict__ b3, float *y, const float *__restrict__ stats, float *out,
                            const float *__restrict__ t, float *dy, float *dZf, __nv_bfloat16 *dZb)
{
    const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (warp >= n) return;
    const float *z = Z2 + (size_t)warp * H;
    float s = 0.f;
#pragma unroll 8
    for (int h = lane; h < H; h += 32) s = fmaf(fmaxf(z[h], 0.f), w3[h], s);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    s = __shfl_sync(0xffffffffu, s, 0) + b3[0];
    if (lane == 0) {
        y[warp] = s;
        if (out) out[warp] = s * stats[1] + stats[0];
    }
    if (!t) return;
    const float r = s - t[warp], d = r / (float)n;
    if (lane == 0) dy[warp] = d;
#pragma unroll 8
    for (int h = lane; h < H; h += 32) {
        const float v = z[h] > 0.f ? d * w3[h] : 0.f;
        dZf[(size_t)warp * H + h] = v;
        dZb[(size_t)warp * H + h] = __float2bfloat16(v);
    }
}

// Adam on FP32 master weights.  The contractions are written out: left to the
// compiler, each kernel's differ in the last bit, and where a gradient is near
// zero the moments' ratio carries that bit into an update of the order of lr.
struct AdamStep {
    float lr, b1, b2, eps, c1, c2;
    __device__ __forceinline__ float operator()(float w, float gi, float &m, float &v) const
    {
        m = fmaf(1.f - b1, gi, b1 * m);
        v = fmaf((1.f - b2) * gi, gi, b2 * v);
        return w - lr * (m / c1) / (sqrtf(v / c2) + eps);
    }
};

// all parameters, then BF16 copies of the two hidden matrices
__global__ void adam_kernel(float *p, const float *__restrict__ g, float *m, float *v, long long n, AdamStep step,
                            __nv_bfloat16 *w1b, long long n_w1, __nv_bfloat16 *w2b, long long off_w2,
                            long long n_w2)
{
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n;
         e += (long long)gridDim.x * blockDim.x) {
        float mi = m[e], vi = v[e];
        const float w = step(p[e], g[e], mi, vi);
        m[e] = mi;
        v[e] = vi;
        p[e] = w;
        if (e < n_w1) w1b[e] = __float2bfloat16(w);
        else if (e >= off_w2 && e < off_w2 + n_w2) w2b[e - off_w2] = __float2bfloat16(w);
    }
}

__global__ void to_bf16_kernel(const float *__restrict__ src, __nv_bfloat16 *dst, long long n)
{
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n;
         e += (long long)gridDim.x * blockDim.x)
        dst[e] = __float2bfloat16(src[e]);
}

// Philox4x32-10 (Salmon et al. 2011) for minibatch sampling
__device__ __forceinline__ uint4 philox_s(uint4 c, uint32_t k0, uint32_t k1)
{
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        if (r) {
            k0 += 0x9E3779B9u;
            k1 += 0xBB67AE85u;
        }
        const uint32_t lo0 = 0xD2511F53u * c.x, hi0 = __umulhi(0xD2511F53u, c.x);
        const uint32_t lo1 = 0xCD9E8D57u * c.z, hi1 = __umulhi(0xCD9E8D57u, c.z);
        c = make_uint4(hi1 ^ c.y ^ k0, lo1, hi0 ^ c.w ^ k1, lo0);
    }
    return c;
}

// Row b of a minibatch of B: drawn uniformly from the filled part of the replay
// buffer (`total` pairs appended so far, `cap` kept); with recent > 0 the second
// half of the batch comes from the newest min(recent, filled) pairs instead (the
// swarm's current neighbourhood).
__device__ __forceinline__ int batch_row(int b, int B, int total, int cap, uint64_t seed, int step, int recent)
{
    const int have = min(total, cap);
    const uint4 w = philox_s(make_uint4((uint32_t)step, (uint32_t)b, 0x5u, 0x7u), (uint32_t)seed,
                             (uint32_t)(seed >> 32));
    if (recent > 0 && b >= B / 2 && have > 0) {
        const int span = min(recent, have);
        const int j = (int)(((unsigned long long)w.x * (unsigned long long)span) >> 32);
        return (int)(((long long)total - 1 - j) % cap);
    }
    return have > 0 ? (int)(((unsigned long long)w.x * (unsigned long long)have) >> 32) : 0;
}

// A minibatch, one warp per row: the drawn row's standardised target (log phi -
// mu) / sigma and its position scaled to [-1, 1] in BF16 (the buffer, of which
// have_host >= 0 pairs are used, else the device's count, holds raw positions).
__global__ void batch_kernel(int B, int K, const int *count, int have_host, int cap, uint64_t seed, int step,
                             int recent, const float *__restrict__ xbuf, const float *__restrict__ ybuf,
                             const float *__restrict__ stats, const double *__restrict__ xmin,
                             const double *__restrict__ xmax, float *t, __nv_bfloat16 *Xb)
{
    const int b = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (b >= B) return;
    const int row = batch_row(b, B, have_host >= 0 ? have_host : *count, cap, seed, step, recent);
    if (lane == 0) t[b] = (ybuf[row] - stats[0]) / stats[1];
    for (int k = lane; k < K; k += 32)
        Xb[(size_t)b * K + k] = normalized(xbuf[(size_t)row * K + k], k, xmin, xmax);
}

// Spearman rank correlation of the k modelled particles' true misfits fk
// and predictions logphi[rows]: ranks by counting (ties by index), one block;
// both keys are staged in shared memory first (k <= 2048)
__global__ void __launch_bounds__(1024)
rank_corr_kernel(const double *__restrict__ fk, const int *__restrict__ rows,
                 const float *__restrict__ logphi, int k, float *rho)
{
    __shared__ double tk[2048];
    __shared__ float pk[2048];
    __shared__ double red[32];
    for (int i = threadIdx.x; i < k; i += blockDim.x) {
        tk[i] = fk[i];
        pk[i] = logphi[rows[i]];
    }
    __syncthreads();
    double d2 = 0.0;
    for (int i = threadIdx.x; i < k; i += blockDim.x) {
        const double ti = tk[i];
        const float pi = pk[i];
        int rt = 0, rp = 0;
        for (int j = 0; j < k; ++j) {
            const double tj = tk[j];
            const float pj = pk[j];
            rt += (tj < ti) || (tj == ti && j < i);
            rp += (pj < pi) || (pj == pi && j < i);
        }
        const double d = (double)(rt - rp);
        d2 += d * d;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) d2 += __shfl_down_sync(0xffffffffu, d2, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = d2;
    __syncthreads();
    if (threadIdx.x == 0) {
        double s = 0.0;
        for (int w = 0; w < (int)blockDim.x / 32; ++w) s += red[w];
        const double kk = (double)k;
        *rho = k > 1 ? (float)(1.0 - 6.0 * s / (kk * (kk * kk - 1.0))) : 1.f;
    }
}

// mean and standard deviation of the filled replay targets, on one cluster of
// STATS_C CTAs (FP64 sums run at 1/64 of the FP32 rate: one CTA took 14 us for
// 6144 targets), summed in a fixed order.  Distributed shared memory may be
// written only once its CTA has started: every CTA arrives at the cluster's
// barrier on entry and waits there before it stores to CTA 0 (the wait falls
// under the sums; with few targets the other CTAs reach their stores at once).
constexpr int STATS_C = 8;
__global__ void __cluster_dims__(STATS_C, 1, 1) __launch_bounds__(512)
stats_kernel(const float *__restrict__ ybuf, const int *count, int have_host, int cap, float *stats)
{
    __shared__ double s1[16], s2[16], c1[STATS_C], c2[STATS_C];
    cooperative_groups::cluster_group cluster = cooperative_groups::this_cluster();
    auto started = cluster.barrier_arrive();
    const int n = min(have_host >= 0 ? have_host : *count, cap);
    double a = 0.0, b = 0.0;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += STATS_C * blockDim.x) {
        const double y = ybuf[i];
        a += y;
        b += y * y;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        a += __shfl_down_sync(0xffffffffu, a, o);
        b += __shfl_down_sync(0xffffffffu, b, o);
    }
    if ((threadIdx.x & 31) == 0) {
        s1[threadIdx.x >> 5] = a;
        s2[threadIdx.x >> 5] = b;
    }
    __syncthreads();
    cluster.barrier_wait(std::move(started));
    if (threadIdx.x == 0) {
        a = b = 0.0;
        for (int w = 0; w < (int)blockDim.x / 32; ++w) {
            a += s1[w];
            b += s2[w];
        }
        *cluster.map_shared_rank(&c1[blockIdx.x], 0) = a;
        *cluster.map_shared_rank(&c2[blockIdx.x], 0) = b;
    }
    cluster.sync();
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        double A = 0.0, Bs = 0.0;
        for (int w = 0; w < STATS_C; ++w) {
            A += c1[w];
            Bs += c2[w];
        }
        double mu = n > 0 ? A / n : 0.0;
        double var = n > 1 ? Bs / n - mu * mu : 1.0;
        stats[0] = (float)mu;
        stats[1] = (float)sqrt(var > 1e-12 ? var : 1e-12);
    }
}

// append (particle, log misfit) pairs; rows with a non-finite misfit are
// skipped.  One block of 1024 threads: the kept rows of each 1024-row chunk
// take consecutive ring slots in row order (an exclusive scan of the keep
// flags), so the buffer order is the same on every run.
__global__ void __launch_bounds__(1024)
append_kernel(const float *__restrict__ x, const double *__restrict__ misfit,
              const int *__restrict__ rows, int n, int K, float *xbuf, float *ybuf, int *count, int cap)
{
    __shared__ int wsum[32];
    __shared__ int slot[1024];
    __shared__ int base, kept;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (tid == 0) base = *count;
    __syncthreads();
    for (int c0 = 0; c0 < n; c0 += 1024) {
        const int m = min(1024, n - c0);
        int ok = 0;
        if (tid < m) {
            const double f = misfit[c0 + tid];
            ok = (isfinite(f) && f > 0.0) ? 1 : 0;
        }
        // inclusive scan within the warp, then over the warp totals
        int v = ok;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int u = __shfl_up_sync(0xffffffffu, v, o);
            if (lane >= o) v += u;
        }
        if (lane == 31) wsum[warp] = v;
        __syncthreads();
        if (warp == 0) {
            int w = wsum[lane];
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int u = __shfl_up_sync(0xffffffffu, w, o);
                if (lane >= o) w += u;
            }
            wsum[lane] = w;   // inclusive totals of warps 0..lane
            if (lane == 31) kept = w;
        }
        __syncthreads();
        const int before = v - ok + (warp > 0 ? wsum[warp - 1] : 0);
        slot[tid] = ok ? (base + before) % cap : -1;
        if (tid < m && ok) ybuf[slot[tid]] = (float)log(misfit[c0 + tid]);
        __syncthreads();
        for (int e = tid; e < m * K; e += blockDim.x) {
            const int i = e / K, kk = e % K;
            const int sl = slot[i];
            if (sl < 0) continue;
            const int src = rows ? rows[c0 + i] : c0 + i;
            xbuf[(size_t)sl * K + kk] = x[(size_t)src * K + kk];
        }
        __syncthreads();
        if (tid == 0) base += kept;
        __syncthreads();
    }
    if (tid == 0) *count = base;
}

// indices of the k smallest keys (ties to the lower index), one block, P <= 2048
__global__ void __launch_bounds__(1024) select_kernel(const float *__restrict__ key, int P, int k, int *out)
{
    __shared__ float kv[2048];
    __shared__ int iv[2048];
    int N = 1;
    while (N < P) N <<= 1;
    for (int i = threadIdx.x; i < N; i += blockDim.x) {
        float v = i < P ? key[i] : __int_as_float(0x7f800000);
        if (!(v == v)) v = __int_as_float(0x7f800000);
        kv[i] = v;
        iv[i] = i < P ? i : 0x7fffffff;
    }
    __syncthreads();
    for (int size = 2; size <= N; size <<= 1)
        for (int stride = size >> 1; stride > 0; stride >>= 1) {
            for (int t = threadIdx.x; t < N / 2; t += blockDim.x) {
                const int lo = 2 * t - (t & (stride - 1)), hi = lo + stride;
                const bool up = (lo & size) == 0;
                const bool lt = kv[hi] < kv[lo] || (kv[hi] == kv[lo] && iv[hi] < iv[lo]);
                const bool gt = kv[lo] < kv[hi] || (kv[lo] == kv[hi] && iv[lo] < iv[hi]);
                if (up ? lt : gt) {
                    const float a = kv[lo];
                    kv[lo] = kv[hi];
                    kv[hi] = a;
                    const int b = iv[lo];
                    iv[lo] = iv[hi];
                    iv[hi] = b;
                }
            }
            __syncthreads();
        }
    for (int i = threadIdx.x; i < k; i += blockDim.x) out[i] = iv[i];
}

// gather selected particles into a compact [k][K] array
__global__ void gather_kernel(const float *__restrict__ x, const int *__restrict__ rows, int k, int K,
                              float *out)
{
    const long long tot = (long long)k * K;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < tot;
         e += (long long)gridDim.x * blockDim.x)
        out[e] = x[(size_t)rows[e / K] * K + e % K];
}

// full-swarm fitness (+inf where not modelled) and EM sort keys (modelled:
// true misfit, others: predicted misfit exp(log phi))
__global__ void scatter_kernel(const int *__restrict__ rows, const double *__restrict__ fk, int k,
                               const float *__restrict__ logphi, int P, double *fit, double *rank)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < P) {
        fit[i] = __longlong_as_double(0x7ff0000000000000LL);
        rank[i] = exp((double)logphi[i]);
    }
}

__global__ void scatter_fill_kernel(const int *__restrict__ rows, const double *__restrict__ fk, int k,
                                    double *fit, double *rank)
{
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j < k) {
        fit[rows[j]] = fk[j];
        rank[rows[j]] = fk[j];
    }
}

// ---------------------------------------------------------------------------
// The whole network in one kernel per 128 batch rows (widths up to 256), for
// which the layers' launches and the trips of Z and A through global memory
// cost more than the products.  rows_kernel: a CTA gathers its rows, keeps both
// weight matrices in shared memory and both accumulators in tensor memory
// (columns 0 .. 255 for layer 1 and again for the data gradient, 256 .. 511 for
// layer 2) and runs X W1 -> A1 W2 -> head; in training also dZ2 -> dZ2 W2 ->
// dZ1, and writes relu(Z2), dZ2 and dZ1 in FP32 for the column sums of the bias
// and head gradients, which grads_kernel takes over the whole batch in the
// layer-by-layer path's order: partial sums per tile (262 us) differ from it in the last
// bit, and Adam turns that into 1e-3 where a gradient is near zero.  A thread owns one
// row and every fourth group of 32 columns; its loops over them stay rolled
// (each line runs once per launch, and unrolled the warps waited for
// instructions).  Six training steps of 1024 pairs and a prediction of 1024, K =
// 32, H = 256: 584 us layer by layer, 281 us here; bound by the latency of the
// chain on 8 CTAs (29 us of a step's kernels under ncu, the gradients 15), with
// the tensor core idle most of it.  grads_kernel: one CTA per 128 x 64
// tile of a weight gradient, fed by bulk copies, with Adam on the tile.
//
// Layout of every matrix in shared memory and of the tiles in global memory
// ("cores"): 8 x 8 BF16 blocks of 128 bytes (8 rows of 16 bytes), block (r / 8,
// c / 8) at ((c / 8) RB + r / 8) 128 with RB the row blocks.  Read as a K-major
// operand (k = c) its core strides are RB 128 along k and 128 along the rows; as
// an MN-major operand (k = r) 128 along k and RB 128 along the columns: one copy
// of W2 serves the forward and the data-gradient product, and a row range of the
// batch tiles is what the weight gradients (k = batch) read, in whole
// contiguous column blocks.
// ---------------------------------------------------------------------------
constexpr int ROWS_THREADS = 512, GRADS_THREADS = 256, HMAX = 256, BT = 128;   // BT: batch rows of a tile

__host__ __device__ inline int up16(int n) { return (n + 15) / 16 * 16; }
__host__ __device__ inline int up32(int n) { return (n + 31) / 32 * 32; }

struct NetArgs {
    int n, K, H;                           // batch rows, inputs, width
    const __nv_bfloat16 *W1b, *W2b;
    const float *b1, *b2, *w3, *b3;
    const double *xmin, *xmax;
    // rows: x[b] of a given batch, or drawn from the replay buffer (sample)
    const float *x, *ybuf, *t;
    int sample, step, recent, have_host, cap;
    const int *count;
    uint64_t seed;
    const float *stats;
    float *out;                            // predictions (no training), log misfit
    // training: tiles [ceil(n / 128)] of X, A1, dZ2, dZ1 in BF16; relu(Z2), dZ2,
    // dZ1 in FP32 [tiles][3][H][128]; dy [tiles][128]; the tiles' losses
    unsigned char *Xt, *A1t, *dZ2t, *dZ1t;
    float *cols, *dy;
    double *part_loss;
    int *err;
};

__device__ __forceinline__ int core_off(int r, int c, int RB)
{
    return ((c >> 3) * RB + (r >> 3)) * 128 + (r & 7) * 16 + (c & 7) * 2;
}

__device__ __forceinline__ void umma(unsigned d, unsigned long long ad, unsigned long long bd, unsigned idesc, bool acc)
{
    asm volatile("{\n .reg .pred p;\n setp.ne.u32 p, %4, 0;\n"
                 " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d),
                 "l"(ad), "l"(bd), "r"(idesc), "r"((unsigned)acc)
                 : "memory");
}
__device__ __forceinline__ void umma_commit(unsigned long long *bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(smem_u32(bar))
                 : "memory");
}

// 32 columns of this thread's row from tensor memory
__device__ __forceinline__ void tmem_row32(unsigned addr, float v[32])
{
    unsigned r[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,"
        "%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];\n"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
          "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
          "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(addr)
        : "memory");
    asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
#pragma unroll
    for (int j = 0; j < 32; ++j) v[j] = __uint_as_float(r[j]);
}

// 8 consecutive values as BF16 into a core row (16 bytes)
__device__ __forceinline__ void store8(unsigned char *dst, const float *v)
{
    __nv_bfloat162 h[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) h[q] = __floats2bfloat162_rn(v[2 * q], v[2 * q + 1]);
    *reinterpret_cast<uint4 *>(dst) = *reinterpret_cast<uint4 *>(h);
}

// rows x cols (a multiple of 8) of a row-major BF16 matrix into cores at dst, by
// asynchronous copies (the columns past `valid`, and odd widths, by plain stores)
__device__ __forceinline__ void load_cores(unsigned char *dst, const __nv_bfloat16 *__restrict__ src, int rows,
                                           int cols, int valid)
{
    const int nv = cols / 8, kg = nv % 4 == 0 ? 4 : 2, per = 8 * kg, bk = nv / kg, RB = rows / 8;
    const bool vec = valid % 8 == 0 && ((size_t)src & 15) == 0;
    for (int v = threadIdx.x; v < rows * nv; v += ROWS_THREADS) {
        const int in = v % per, blk = v / per;
        const int r = (blk / bk) * 8 + (in & 7), c = ((blk % bk) * kg + (in >> 3)) * 8;
        unsigned char *d = dst + core_off(r, c, RB);
        if (vec && c < valid) {
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(smem_u32(d)), "l"(src + (size_t)r * valid + c)
                         : "memory");
        } else {
            __nv_bfloat16 t[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) t[e] = c + e < valid ? src[(size_t)r * valid + c + e] : __float2bfloat16(0.f);
            *reinterpret_cast<uint4 *>(d) = *reinterpret_cast<const uint4 *>(t);
        }
    }
}

// shared-memory plan of rows_kernel (bytes): W2, the A1 / dZ2 / dZ1 tile, then X
// and W1 when they fit
// beside, else X in the tile's place and W1 in W2's until layer 1 is done
struct RowsPlan {
    int w2, tile, x, w1, vec, bytes;
    bool beside;
};
__host__ __device__ inline RowsPlan rows_plan(int K, int H)
{
    const int Kp = up16(K), xb = BT * Kp * 2, w1b = H * Kp * 2;
    const int vecb = (3 * up32(H) + 2 * Kp + 2 * BT + HMAX / 32 * BT) * 4;
    RowsPlan p{};
    p.w2 = 0;
    p.tile = H * H * 2;
    const int end = p.tile + BT * H * 2, most = 227 * 1024 - 1024;
    p.beside = end + xb + w1b + vecb <= most;
    if (p.beside) {
        p.x = end;
        p.w1 = end + xb;
        p.vec = p.w1 + w1b;
    } else {
        // room for X and W1 where W2 and the tile will be
        const int tile = p.tile > w1b ? p.tile : w1b;
        p.tile = tile;
        p.x = tile;
        p.w1 = 0;
        p.vec = tile + (BT * H * 2 > xb ? BT * H * 2 : xb);
    }
    p.bytes = p.vec + vecb;
    return p;
}

template <bool TRAIN>
__global__ void __launch_bounds__(ROWS_THREADS, 1) rows_kernel(const NetArgs a)
{
    extern __shared__ __align__(1024) unsigned char tsm[];
    __shared__ __align__(8) unsigned long long mbar;
    __shared__ unsigned tmem_base;
    __shared__ int s_fail;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int K = a.K, H = a.H, Kp = up16(K), b0 = blockIdx.x * BT, tile = blockIdx.x;
    const RowsPlan pl = rows_plan(K, H);
    unsigned char *W2s = tsm + pl.w2, *T = tsm + pl.tile, *Xs = tsm + pl.x, *W1s = tsm + pl.w1;
    float *vec = reinterpret_cast<float *>(tsm + pl.vec);
    const int Hp = up32(H);                 // the vectors are zero past H
    float *b1 = vec, *b2 = vec + Hp, *w3 = vec + 2 * Hp, *lo = vec + 3 * Hp, *hi = lo + Kp, *ts = hi + Kp, *dys = ts + BT;
    unsigned *on = reinterpret_cast<unsigned *>(dys + BT);       // signs of A1: [group of 32 columns][row]
    if (tid == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(smem_u32(&mbar)) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
        s_fail = 0;
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_u32(&tmem_base)),
                     "r"(512u)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
    }
    load_cores(W1s, a.W1b, H, Kp, K);
    asm volatile("cp.async.commit_group;\n" ::: "memory");
    if (pl.beside) load_cores(W2s, a.W2b, H, H, H);
    asm volatile("cp.async.commit_group;\n" ::: "memory");
    for (int h = tid; h < Hp; h += ROWS_THREADS) {
        b1[h] = h < H ? a.b1[h] : 0.f;
        b2[h] = h < H ? a.b2[h] : 0.f;
        w3[h] = h < H ? a.w3[h] : 0.f;
    }
    for (int k = tid; k < K; k += ROWS_THREADS) {
        lo[k] = (float)a.xmin[k];
        hi[k] = (float)a.xmax[k];
    }
    __syncthreads();
    // X: 16 rows per warp, scaled to [-1, 1]; zeros past the batch and the inputs
    {
        const int total = TRAIN && a.sample ? (a.have_host >= 0 ? a.have_host : *a.count) : 0;
        constexpr int RW = BT / (ROWS_THREADS / 32);       // rows of a warp; lane i draws row i
        const int bl = b0 + warp * RW + lane;
        int row_l = bl;
        float t_l = 0.f;
        if (lane < RW && bl < a.n && TRAIN) {
            if (a.sample) {
                row_l = batch_row(bl, a.n, total, a.cap, a.seed, a.step, a.recent);
                t_l = (a.ybuf[row_l] - a.stats[0]) / a.stats[1];
            } else {
                t_l = a.t[bl];
            }
        }
        if (lane < RW) ts[warp * RW + lane] = t_l;
#pragma unroll 4
        for (int i = 0; i < RW; ++i) {
            const int r = warp * RW + i, row = __shfl_sync(0xffffffffu, row_l, i);
            for (int k = lane; k < Kp; k += 32) {
                float v = 0.f;
                if (b0 + r < a.n && k < K) v = 2.f * (a.x[(size_t)row * K + k] - lo[k]) / (hi[k] - lo[k]) - 1.f;
                *reinterpret_cast<__nv_bfloat16 *>(Xs + core_off(r, k, BT / 8)) = __float2bfloat16(v);
            }
        }
    }
    asm volatile("cp.async.wait_group 1;\n" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    const unsigned tmem = tmem_base, idesc = umma_idesc(BT, H);
    unsigned parity = 0;
    // waits for the products issued last (bounded; gives up once)
    auto products = [&] {
        if (!mbar_wait_tc(smem_u32(&mbar), parity)) s_fail = 1;
        parity ^= 1;
        asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    };
    // a tile in shared memory to global memory (thread 0; its reads are awaited
    // before the place is written again)
    auto bulk_out = [&](unsigned char *dst, const unsigned char *src, unsigned bytes) {
        asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;\n" ::"l"(dst), "r"(smem_u32(src)),
                     "r"(bytes)
                     : "memory");
        asm volatile("cp.async.bulk.commit_group;\n" ::: "memory");
    };
    auto bulk_read = [] { asm volatile("cp.async.bulk.wait_group.read 0;\n" ::: "memory"); };
    if (tid == 0) {
        for (int s = 0; s < Kp / 16; ++s)
            umma(tmem, umma_desc(Xs + s * 2 * (BT / 8) * 128, BT / 8 * 128, 128),
                 umma_desc(W1s + s * 2 * (H / 8) * 128, H / 8 * 128, 128), idesc, s > 0);
        umma_commit(&mbar);
        if (TRAIN) bulk_out(a.Xt + (size_t)tile * BT * Kp * 2, Xs, BT * Kp * 2);
    }
    products();
    if (!pl.beside) {
        if (TRAIN && tid == 0) bulk_read();        // X's place becomes the tile's
        __syncthreads();
        load_cores(W2s, a.W2b, H, H, H);
    }
    asm volatile("cp.async.commit_group;\n" ::: "memory");
    // layer 1: A1 = relu(Z1 + b1) as the next product's operand; the signs are
    // kept for the way back
    const int r = 32 * (warp & 3) + lane, part = warp >> 2;
    constexpr int STEP = 32 * (ROWS_THREADS / 128);      // columns from one group of a thread to its next
    const bool real = b0 + r < a.n;
    const unsigned trow = tmem + ((unsigned)(32 * (warp & 3)) << 16);
#pragma unroll 1
    for (int c0 = 32 * part; c0 < H; c0 += STEP) {
        float v[32];
        tmem_row32(trow + c0, v);
        unsigned bits = 0u;
#pragma unroll
        for (int j = 0; j < 32; j += 4) {                // (columns past H go nowhere)
            const float4 b = *reinterpret_cast<const float4 *>(b1 + c0 + j);
            v[j] = fmaxf(v[j] + b.x, 0.f);
            v[j + 1] = fmaxf(v[j + 1] + b.y, 0.f);
            v[j + 2] = fmaxf(v[j + 2] + b.z, 0.f);
            v[j + 3] = fmaxf(v[j + 3] + b.w, 0.f);
        }
        if (TRAIN) {
#pragma unroll
            for (int j = 0; j < 32; ++j) bits |= v[j] > 0.f ? 1u << j : 0u;
        }
        if (TRAIN) on[c0 / 32 * BT + r] = bits;
#pragma unroll
        for (int j = 0; j < 32; j += 8)
            if (c0 + j < H) store8(T + core_off(r, c0 + j, BT / 8), v + j);
    }
    asm volatile("cp.async.wait_group 0;\n" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    if (tid == 0) {
        asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
        for (int s = 0; s < H / 16; ++s)
            umma(tmem + HMAX, umma_desc(T + s * 2 * (BT / 8) * 128, BT / 8 * 128, 128),
                 umma_desc(W2s + s * 2 * (H / 8) * 128, H / 8 * 128, 128), idesc, s > 0);
        umma_commit(&mbar);
        if (TRAIN) bulk_out(a.A1t + (size_t)tile * BT * H * 2, T, BT * H * 2);
    }
    products();
    // head: y = sum_h relu(Z2) w3 + b3 in the order of 32 strided partial sums
    // added pairwise (one thread per row)
    if (part == 0) {
        float s[32];
#pragma unroll
        for (int j = 0; j < 32; ++j) s[j] = 0.f;
#pragma unroll 1
        for (int c0 = 0; c0 < H; c0 += 32) {
            float v[32];
            tmem_row32(trow + HMAX + c0, v);
#pragma unroll
            for (int j = 0; j < 32; j += 16) {           // (H is a multiple of 16)
                if (c0 + j >= H) break;
#pragma unroll
                for (int i = j; i < j + 16; i += 4) {
                    const float4 b = *reinterpret_cast<const float4 *>(b2 + c0 + i);
                    const float4 w = *reinterpret_cast<const float4 *>(w3 + c0 + i);
                    s[i] = fmaf(fmaxf(v[i] + b.x, 0.f), w.x, s[i]);
                    s[i + 1] = fmaf(fmaxf(v[i + 1] + b.y, 0.f), w.y, s[i + 1]);
                    s[i + 2] = fmaf(fmaxf(v[i + 2] + b.z, 0.f), w.z, s[i + 2]);
                    s[i + 3] = fmaf(fmaxf(v[i + 3] + b.w, 0.f), w.w, s[i + 3]);
                }
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
#pragma unroll
            for (int j = 0; j < o; ++j) s[j] += s[j + o];
        const float y = s[0] + a.b3[0];
        if (!TRAIN) {
            if (real) a.out[b0 + r] = y * a.stats[1] + a.stats[0];
        } else {
            const float e = y - ts[r];
            dys[r] = real ? e / (float)a.n : 0.f;
            ts[r] = real ? e : 0.f;
        }
    }
    if (TRAIN) {
        if (tid == 0) bulk_read();                 // A1 has left the tile
        __syncthreads();
        if (warp == ROWS_THREADS / 32 - 1) {       // the tile's loss (fixed order)
            double sl = 0.0;
            for (int i = lane; i < BT; i += 32) sl += (double)ts[i] * ts[i];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) sl += __shfl_down_sync(0xffffffffu, sl, o);
            if (lane == 0) a.part_loss[tile] = sl;
        }
        if (part == 0) a.dy[(size_t)tile * BT + r] = dys[r];
        // what grads_kernel sums over the batch: relu(Z2), dZ2, dZ1 in FP32, a column's
        // rows side by side
        float *const col = a.cols + (size_t)tile * 3 * H * BT + r;
        auto keep = [&](int q, int c0, const float v[32]) {
#pragma unroll
            for (int j = 0; j < 32; j += 16) {           // (H is a multiple of 16)
                if (c0 + j >= H) break;
#pragma unroll
                for (int i = j; i < j + 16; ++i) col[(size_t)(q * H + c0 + i) * BT] = v[i];
            }
        };
        // dZ2 = dy w3 [Z2 > 0]
        const float dy = dys[r];
#pragma unroll 1
        for (int c0 = 32 * part; c0 < H; c0 += STEP) {
            float v[32], z[32];
            tmem_row32(trow + HMAX + c0, z);
#pragma unroll
            for (int j = 0; j < 32; j += 4) {            // (columns past H go nowhere)
                const float4 b = *reinterpret_cast<const float4 *>(b2 + c0 + j);
                const float4 w = *reinterpret_cast<const float4 *>(w3 + c0 + j);
                auto one = [&](int i, float bb, float ww) {
                    const float zz = z[i] + bb;
                    v[i] = zz > 0.f && real ? dy * ww : 0.f;
                    z[i] = real ? fmaxf(zz, 0.f) : 0.f;
                };
                one(j, b.x, w.x);
                one(j + 1, b.y, w.y);
                one(j + 2, b.z, w.z);
                one(j + 3, b.w, w.w);
            }
#pragma unroll
            for (int j = 0; j < 32; j += 8)
                if (c0 + j < H) store8(T + core_off(r, c0 + j, BT / 8), v + j);
            keep(0, c0, z);
            keep(1, c0, v);
        }
        asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
        asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
        __syncthreads();
        if (tid == 0) {
            asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
            // dA1 = dZ2 W2: W2 read MN-major (k = its rows)
            for (int s = 0; s < H / 16; ++s)
                umma(tmem, umma_desc(T + s * 2 * (BT / 8) * 128, BT / 8 * 128, 128),
                     umma_desc(W2s + s * 2 * 128, 128, H / 8 * 128), idesc | (1u << 16), s > 0);
            umma_commit(&mbar);
            bulk_out(a.dZ2t + (size_t)tile * BT * H * 2, T, BT * H * 2);
        }
        products();
        if (tid == 0) bulk_read();                 // dZ2 has left the tile
        __syncthreads();
#pragma unroll 1
        for (int c0 = 32 * part; c0 < H; c0 += STEP) {
            float v[32];
            tmem_row32(trow + c0, v);
            const unsigned bits = real ? on[c0 / 32 * BT + r] : 0u;
#pragma unroll
            for (int j = 0; j < 32; ++j) v[j] = (bits >> j & 1u) ? v[j] : 0.f;
#pragma unroll
            for (int j = 0; j < 32; j += 8)
                if (c0 + j < H) store8(T + core_off(r, c0 + j, BT / 8), v + j);
            keep(2, c0, v);
        }
        asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
        asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
        __syncthreads();
        if (tid == 0) bulk_out(a.dZ1t + (size_t)tile * BT * H * 2, T, BT * H * 2);
    }
    if (tid == 0) {
        asm volatile("cp.async.bulk.wait_group 0;\n" ::: "memory");   // every tile is written
        if (s_fail) atomicExch(a.err, EMPSO_TIMEOUT);
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(512u) : "memory");
}

// Weight gradients of `tiles` batch tiles: the CTAs of g_W2 (128 x 64 tiles of
// dZ2^T A1), of g_W1 (dZ1^T X), and those of the vectors.  The batch tiles come
// in by bulk copies, GSTAGES in flight (a tile's columns are contiguous
// blocks); the accumulator takes them in batch order.  With `adam` the
// gradient's tile is applied at once, else it is written.
constexpr int GT_N = 64, GSTAGES = 4, GA_BYTES = 128 * BT * 2, GB_BYTES = GT_N * BT * 2;
constexpr int GRADS_SMEM = GSTAGES * (GA_BYTES + GB_BYTES);

struct GradArgs {
    int n, tiles, K, H, adam;
    const unsigned char *Xt, *A1t, *dZ2t, *dZ1t;
    const float *cols, *dy;
    const double *part_loss;
    float *p, *g, *m, *v, *loss;
    long long off_b1, off_W2, off_b2, off_w3, off_b3;
    __nv_bfloat16 *W1b, *W2b;
    AdamStep step;
    int *err;
};

__device__ __forceinline__ void apply_grad(const GradArgs &a, long long e, float gi, __nv_bfloat16 *wb)
{
    if (!a.adam) {
        a.g[e] = gi;
        return;
    }
    float m = a.m[e], v = a.v[e];
    const float w = a.step(a.p[e], gi, m, v);
    a.m[e] = m;
    a.v[e] = v;
    a.p[e] = w;
    if (wb) *wb = __float2bfloat16(w);
}

constexpr int SUM_COLS = 4;              // columns of a warp of the vectors' CTAs
__host__ __device__ inline int vector_ctas(int H) { return 1 + (3 * H + GRADS_THREADS / 32 * SUM_COLS - 1) / (GRADS_THREADS / 32 * SUM_COLS); }
__host__ __device__ inline int grad_tiles(int H, int N) { return (H + 127) / 128 * ((N + GT_N - 1) / GT_N); }

__global__ void __launch_bounds__(GRADS_THREADS, 1) grads_kernel(const GradArgs a)
{
    extern __shared__ __align__(1024) unsigned char tsm[];
    __shared__ __align__(8) unsigned long long full[GSTAGES], done[GSTAGES];
    __shared__ unsigned tmem_base;
    __shared__ int s_fail;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, H = a.H, Kp = up16(a.K);
    const int n2 = grad_tiles(H, H), n1 = grad_tiles(H, Kp);
    int b = blockIdx.x;
    if (b >= n2 + n1) {
        b -= n2 + n1;
        if (b == 0) {                                    // b3 and the loss
            float s = 0.f;
            sum_all(a.dy, a.n, &s);
            if (tid == 0) {
                apply_grad(a, a.off_b3, s, nullptr);
                double l = 0.0;
                for (int t = 0; t < a.tiles; ++t) l += a.part_loss[t];
                if (a.loss) *a.loss = (float)(0.5 * l / a.n);
            }
            return;
        }
        // w3, b2, b1: a warp per SUM_COLS columns; lane i adds rows i, i + 32, ..,
        // then the lanes' sums are added pairwise (the order of the layer-by-layer path)
        const int e0 = ((b - 1) * (GRADS_THREADS / 32) + warp) * SUM_COLS;
        float s[SUM_COLS];
        const float *src[SUM_COLS];
#pragma unroll
        for (int i = 0; i < SUM_COLS; ++i) {
            s[i] = 0.f;
            src[i] = a.cols + (size_t)min(e0 + i, 3 * H - 1) * BT + lane;
        }
        for (int t = 0; t < a.tiles; ++t)
#pragma unroll
            for (int k = 0; k < BT; k += 32) {
                const float dy = a.dy[t * BT + k + lane];
#pragma unroll
                for (int i = 0; i < SUM_COLS; ++i) {
                    const float v = src[i][(size_t)t * 3 * H * BT + k];
                    s[i] = e0 + i < H ? fmaf(v, dy, s[i]) : s[i] + v;
                }
            }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
#pragma unroll
            for (int i = 0; i < SUM_COLS; ++i) s[i] += __shfl_down_sync(0xffffffffu, s[i], o);
        if (lane == 0)
#pragma unroll
            for (int i = 0; i < SUM_COLS; ++i) {
                const int e = e0 + i, q = e / H, h = e % H;
                if (e < 3 * H) apply_grad(a, (q == 0 ? a.off_w3 : (q == 1 ? a.off_b2 : a.off_b1)) + h, s[i], nullptr);
            }
        return;
    }
    const bool second = b < n2;
    if (!second) b -= n2;
    const int N = second ? H : Kp, Nv = second ? H : a.K;          // columns staged, columns that exist
    const int nx = (N + GT_N - 1) / GT_N, m0 = b / nx * 128, n0 = b % nx * GT_N;
    const int mc = min(128, H - m0), nc = min(GT_N, N - n0);
    const unsigned char *At = second ? a.dZ2t : a.dZ1t, *Bt = second ? a.A1t : a.Xt;
    const size_t a_tile = (size_t)BT * H * 2, b_tile = (size_t)BT * N * 2;
    const size_t a_ofs = (size_t)(m0 / 8) * (BT / 8) * 128, b_ofs = (size_t)(n0 / 8) * (BT / 8) * 128;
    const unsigned a_bytes = mc * BT * 2, b_bytes = nc * BT * 2;
    if (tid == 0) {
        for (int i = 0; i < GSTAGES; ++i) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(smem_u32(&full[i])) : "memory");
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(smem_u32(&done[i])) : "memory");
        }
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
        s_fail = 0;
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_u32(&tmem_base)),
                     "r"(64u)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    const unsigned tmem = tmem_base;
    if (tid == 0) {
        const unsigned idesc = umma_idesc(128, nc) | (1u << 15) | (1u << 16);     // both MN-major (k = batch row)
        auto fetch = [&](int t) {
            const int st = t % GSTAGES;
            unsigned char *As = tsm + st * (GA_BYTES + GB_BYTES), *Bs = As + GA_BYTES;
            asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(smem_u32(&full[st])),
                         "r"(a_bytes + b_bytes)
                         : "memory");
            asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n" ::"r"(
                             smem_u32(As)),
                         "l"(At + t * a_tile + a_ofs), "r"(a_bytes), "r"(smem_u32(&full[st]))
                         : "memory");
            asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n" ::"r"(
                             smem_u32(Bs)),
                         "l"(Bt + t * b_tile + b_ofs), "r"(b_bytes), "r"(smem_u32(&full[st]))
                         : "memory");
        };
        for (int t = 0; t < min(a.tiles, GSTAGES); ++t) fetch(t);
        for (int t = 0; t < a.tiles; ++t) {
            const int st = t % GSTAGES;
            unsigned char *As = tsm + st * (GA_BYTES + GB_BYTES), *Bs = As + GA_BYTES;
            if (!mbar_wait_tc(smem_u32(&full[st]), (t / GSTAGES) & 1)) s_fail = 1;
            asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
            for (int s = 0; s < BT / 16; ++s)
                umma(tmem, umma_desc(As + s * 2 * 128, 128, BT / 8 * 128), umma_desc(Bs + s * 2 * 128, 128, BT / 8 * 128),
                     idesc, t > 0 || s > 0);
            umma_commit(&done[st]);
            // the stage of the tile before this one takes the tile after next
            const int f = t - 1 + GSTAGES;
            if (t >= 1 && f < a.tiles) {
                if (!mbar_wait_tc(smem_u32(&done[(t - 1) % GSTAGES]), ((t - 1) / GSTAGES) & 1)) s_fail = 1;
                fetch(f);
            }
        }
        const int t = a.tiles - 1;                 // the last commit covers every product before it
        if (!mbar_wait_tc(smem_u32(&done[t % GSTAGES]), (t / GSTAGES) & 1)) s_fail = 1;
        // a wait that gave up may have left its copies in flight: they are waited for
        // once more (bounded) before the CTA gives its shared memory back
        if (s_fail)
            for (int i = max(0, a.tiles - GSTAGES); i < a.tiles; ++i)
                mbar_wait_tc(smem_u32(&full[i % GSTAGES]), (i / GSTAGES) & 1);
    }
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    // the tile through shared memory, so that parameters are read and written in rows
    constexpr int GP = GT_N + 4;
    float *G = reinterpret_cast<float *>(tsm);
    for (int c0 = 32 * (warp >> 2); c0 < GT_N; c0 += 64) {
        float v[32];
        tmem_row32(tmem + ((unsigned)(32 * (warp & 3)) << 16) + c0, v);
#pragma unroll
        for (int j = 0; j < 32; j += 4)
            *reinterpret_cast<float4 *>(G + (32 * (warp & 3) + lane) * GP + c0 + j) =
                make_float4(v[j], v[j + 1], v[j + 2], v[j + 3]);
    }
    __syncthreads();
    const long long off = second ? a.off_W2 : 0;
    __nv_bfloat16 *Wb = second ? a.W2b : a.W1b;
    if (!s_fail && a.adam && Nv % 4 == 0 && off % 4 == 0) {
        // four parameters at a time, the loads of four such groups together
        constexpr int Q = GT_N / 4, IT = 128 * Q / GRADS_THREADS, UN = 4;
        for (int i0 = 0; i0 < IT; i0 += UN) {
            float4 p[UN], m[UN], v[UN];
            long long q[UN];
            bool on[UN];
#pragma unroll
            for (int i = 0; i < UN; ++i) {
                const int e = tid + (i0 + i) * GRADS_THREADS, r = e / Q, c = e % Q * 4;
                on[i] = r < mc && n0 + c < Nv && c < nc;
                q[i] = (long long)(m0 + r) * Nv + n0 + c;
                if (on[i]) {
                    p[i] = *reinterpret_cast<const float4 *>(a.p + off + q[i]);
                    m[i] = *reinterpret_cast<const float4 *>(a.m + off + q[i]);
                    v[i] = *reinterpret_cast<const float4 *>(a.v + off + q[i]);
                }
            }
#pragma unroll
            for (int i = 0; i < UN; ++i) {
                if (!on[i]) continue;
                const int e = tid + (i0 + i) * GRADS_THREADS, r = e / Q, c = e % Q * 4;
                const float4 gi = *reinterpret_cast<const float4 *>(G + r * GP + c);
                p[i].x = a.step(p[i].x, gi.x, m[i].x, v[i].x);
                p[i].y = a.step(p[i].y, gi.y, m[i].y, v[i].y);
                p[i].z = a.step(p[i].z, gi.z, m[i].z, v[i].z);
                p[i].w = a.step(p[i].w, gi.w, m[i].w, v[i].w);
                *reinterpret_cast<float4 *>(a.p + off + q[i]) = p[i];
                *reinterpret_cast<float4 *>(a.m + off + q[i]) = m[i];
                *reinterpret_cast<float4 *>(a.v + off + q[i]) = v[i];
                const __nv_bfloat162 h0 = __floats2bfloat162_rn(p[i].x, p[i].y), h1 = __floats2bfloat162_rn(p[i].z, p[i].w);
                reinterpret_cast<__nv_bfloat162 *>(Wb + q[i])[0] = h0;
                reinterpret_cast<__nv_bfloat162 *>(Wb + q[i])[1] = h1;
            }
        }
    } else if (!s_fail) {
        for (int e = tid; e < 128 * GT_N; e += GRADS_THREADS) {
            const int r = e / GT_N, c = e % GT_N;
            if (r >= mc || n0 + c >= Nv || c >= nc) continue;
            const long long q = (long long)(m0 + r) * Nv + n0 + c;
            apply_grad(a, off + q, G[r * GP + c], Wb + q);
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(64u) : "memory");
    if (tid == 0 && s_fail) atomicExch(a.err, EMPSO_TIMEOUT);
}

inline int blocks_for(long long n, int per = 256)
{
    long long b = (n + per - 1) / per;
    return (int)(b < 1 ? 1 : (b > 4096 ? 4096 : b));
}

}  // namespace

// ---------------------------------------------------------------------------
// host-side launchers used by api.cu
// ---------------------------------------------------------------------------

// opt the tcgen05 kernels into their shared memory (current device)
cudaError_t sur_prepare_tc(const SurDev &)
{
    cudaError_t e = cudaFuncSetAttribute(jobs_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, TC_SMEM);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(grads_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, GRADS_SMEM);
    // (the largest plan: the attribute is the kernel's, not the network's)
    constexpr int MOST = 227 * 1024 - 1024;
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(rows_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, MOST);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(rows_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, MOST);
    return e;
}

// does the whole-network kernel take this network (and backend)?
bool sur_whole(const SurDev &s)
{
    return s.tc && s.err && s.H <= HMAX && up16(s.K) <= HMAX && rows_plan(s.K, s.H).bytes <= 227 * 1024 - 1024;
}

// bytes of one batch tile's X, A1, dZ2 and dZ1 and its partial sums
size_t sur_tile_bytes(int K, int H) { return (size_t)BT * (up16(K) + 3 * H) * 2 + 12 * (size_t)H * BT + 4 * BT + 8; }

namespace {

// both hidden layers of batch Xb [n][K]: A1b = relu(X W1 + b1) (BF16), Z2
cudaError_t hidden_layers(const SurDev &s, const __nv_bfloat16 *Xb, int n, cudaStream_t st)
{
    cudaError_t e;
    if ((e = run_gemm(s, {n, s.H, s.K, Xb, s.K, 1, s.W1b, s.K, 1, s.p + s.off_b1, 1, nullptr, 0, nullptr, 0, s.A1b, s.H}, st)))
        return e;
    return run_gemm(s, {n, s.H, s.H, s.A1b, s.H, 1, s.W2b, s.H, 1, s.p + s.off_b2, 0, nullptr, 0, s.Z2, s.H, nullptr, 0}, st);
}

}  // namespace

namespace {

AdamStep adam_step(SurDev &s)
{
    s.t += 1;
    return {s.lr, s.beta1, s.beta2, s.eps, 1.f - powf(s.beta1, (float)s.t), 1.f - powf(s.beta2, (float)s.t)};
}

NetArgs net_args(const SurDev &s, int n)
{
    NetArgs a{};
    a.n = n;
    a.K = s.K;
    a.H = s.H;
    a.W1b = s.W1b;
    a.W2b = s.W2b;
    a.b1 = s.p + s.off_b1;
    a.b2 = s.p + s.off_b2;
    a.w3 = s.p + s.off_w3;
    a.b3 = s.p + s.off_b3;
    a.xmin = s.xmin;
    a.xmax = s.xmax;
    a.stats = s.stats;
    a.err = s.err;
    return a;
}

// forward, backward and (step given) the update, two launches; the rows of `a`
// are set.  The tiles lie one kind after the other in s.tiles.
cudaError_t whole_step(const SurDev &s, NetArgs a, const AdamStep *step, float *loss, cudaStream_t st)
{
    const int T = (a.n + BT - 1) / BT, Kp = up16(s.K);
    unsigned char *q = s.tiles;
    auto take = [&](size_t bytes) {
        unsigned char *p = q;
        q += bytes * T;
        return p;
    };
    a.Xt = take((size_t)BT * Kp * 2);
    a.A1t = take((size_t)BT * s.H * 2);
    a.dZ2t = take((size_t)BT * s.H * 2);
    a.dZ1t = take((size_t)BT * s.H * 2);
    a.part_loss = reinterpret_cast<double *>(take(8));
    a.cols = reinterpret_cast<float *>(take(12 * (size_t)s.H * BT));
    a.dy = reinterpret_cast<float *>(take(4 * BT));
    rows_kernel<true><<<T, ROWS_THREADS, rows_plan(s.K, s.H).bytes, st>>>(a);
    GradArgs g{};
    g.n = a.n;
    g.tiles = T;
    g.K = s.K;
    g.H = s.H;
    g.adam = step != nullptr;
    if (step) g.step = *step;
    g.Xt = a.Xt;
    g.A1t = a.A1t;
    g.dZ2t = a.dZ2t;
    g.dZ1t = a.dZ1t;
    g.cols = a.cols;
    g.dy = a.dy;
    g.part_loss = a.part_loss;
    g.p = s.p;
    g.g = s.g;
    g.m = s.m;
    g.v = s.v;
    g.loss = loss;
    g.off_b1 = s.off_b1;
    g.off_W2 = s.off_W2;
    g.off_b2 = s.off_b2;
    g.off_w3 = s.off_w3;
    g.off_b3 = s.off_b3;
    g.W1b = s.W1b;
    g.W2b = s.W2b;
    g.err = s.err;
    grads_kernel<<<grad_tiles(s.H, s.H) + grad_tiles(s.H, Kp) + vector_ctas(s.H), GRADS_THREADS, GRADS_SMEM, st>>>(g);
    return cudaGetLastError();
}

}  // namespace

// gradient of the half-MSE on batch (x [n][K] positions, t [n]) into s.g; loss
// to *loss (device float, may be null)
cudaError_t sur_gradient(const SurDev &s, const float *x, const float *t, int n, float *loss, cudaStream_t st)
{
    if (sur_whole(s)) {
        NetArgs a = net_args(s, n);
        a.x = x;
        a.t = t;
        return whole_step(s, a, nullptr, loss, st);
    }
    cudaError_t e = sur_normalize(s, x, n, s.Xb, st);
    return e ? e : sur_backward(s, s.Xb, t, n, loss, st);
}

// the same from BF16 rows, layer by layer
cudaError_t sur_backward(const SurDev &s, const __nv_bfloat16 *Xb, const float *t, int n,
                         float *loss, cudaStream_t st)
{
    cudaError_t e;
    if ((e = hidden_layers(s, Xb, n, st))) return e;
    head_kernel<<<(n * 32 + 255) / 256, 256, 0, st>>>(s.Z2, n, s.H, s.p + s.off_w3, s.p + s.off_b3, s.y, nullptr,
                                                      nullptr, t, s.dy, s.dZf, s.dZb);
    // dZ1 = (dZ2 W2) [A1 > 0]; g_W2[h][h'] = sum_b dZ2[b][h] A1[b][h']; the
    // head's g_w3 = sum_b relu(Z2) dy and g_b3 = sum_b dy; g_b2; the loss
    Jobs j;
    j.n_gemm = 2;
    j.g[0] = {s.H, s.H, n, s.dZb, s.H, 0, s.A1b, s.H, 0, nullptr, 0, nullptr, 0, s.g + s.off_W2, s.H, nullptr, 0};
    j.g[1] = {n, s.H, s.H, s.dZb, s.H, 1, s.W2b, s.H, 0, nullptr, 0, s.A1b, s.H, s.dA, s.H, s.dZ1b, s.H};
    j.n_col = 2;
    j.c[0] = {s.Z2, s.dy, n, s.H, s.g + s.off_w3};
    j.c[1] = {s.dZf, nullptr, n, s.H, s.g + s.off_b2};
    j.sums = 1;
    j.dy = s.dy;
    j.y = s.y;
    j.t = t;
    j.n = n;
    j.gb3 = s.g + s.off_b3;
    j.loss = loss;
    if ((e = run_jobs(s, j, st))) return e;
    // g_W1[h][k] = sum_b dZ1[b][h] X[b][k]; g_b1
    Jobs i;
    i.n_gemm = 1;
    i.g[0] = {s.H, s.K, n, s.dZ1b, s.H, 0, Xb, s.K, 0, nullptr, 0, nullptr, 0, s.g + s.off_W1, s.K, nullptr, 0};
    i.n_col = 1;
    i.c[0] = {s.dA, nullptr, n, s.H, s.g + s.off_b1};
    return run_jobs(s, i, st);
}

cudaError_t sur_adam(SurDev &s, cudaStream_t st)
{
    adam_kernel<<<blocks_for(s.n_params), 256, 0, st>>>(s.p, s.g, s.m, s.v, s.n_params, adam_step(s), s.W1b,
                                                        (long long)s.H * s.K, s.W2b, s.off_W2,
                                                        (long long)s.H * s.H);
    return cudaGetLastError();
}

cudaError_t sur_refresh_bf16(const SurDev &s, cudaStream_t st)
{
    to_bf16_kernel<<<blocks_for((long long)s.H * s.K), 256, 0, st>>>(s.p + s.off_W1, s.W1b,
                                                                     (long long)s.H * s.K);
    to_bf16_kernel<<<blocks_for((long long)s.H * s.H), 256, 0, st>>>(s.p + s.off_W2, s.W2b,
                                                                     (long long)s.H * s.H);
    return cudaGetLastError();
}

cudaError_t sur_normalize(const SurDev &s, const float *x, int n, __nv_bfloat16 *out, cudaStream_t st)
{
    normalize_kernel<<<blocks_for((long long)n * s.K), 256, 0, st>>>(x, n, s.K, s.xmin, s.xmax, out);
    return cudaGetLastError();
}

cudaError_t sur_predict(const SurDev &s, const float *x, int n, float *logphi, cudaStream_t st)
{
    if (sur_whole(s)) {
        NetArgs a = net_args(s, n);
        a.x = x;
        a.out = logphi;
        rows_kernel<false><<<(n + BT - 1) / BT, ROWS_THREADS, rows_plan(s.K, s.H).bytes, st>>>(a);
        return cudaGetLastError();
    }
    cudaError_t e;
    if ((e = sur_normalize(s, x, n, s.Xb, st))) return e;
    if ((e = hidden_layers(s, s.Xb, n, st))) return e;
    head_kernel<<<(n * 32 + 255) / 256, 256, 0, st>>>(s.Z2, n, s.H, s.p + s.off_w3, s.p + s.off_b3, s.y, s.stats,
                                                      logphi, nullptr, nullptr, nullptr, nullptr);
    return cudaGetLastError();
}

cudaError_t sur_append(const SurDev &s, const float *x, const double *misfit, const int *rows, int n,
                       cudaStream_t st)
{
    append_kernel<<<1, 1024, 0, st>>>(x, misfit, rows, n, s.K, s.xbuf, s.ybuf, s.count, s.cap);
    return cudaGetLastError();
}

cudaError_t sur_train(SurDev &s, int steps, int B, cudaStream_t st, int have)
{
    cudaError_t e;
    stats_kernel<<<STATS_C, 512, 0, st>>>(s.ybuf, s.count, have, s.cap, s.stats);
    for (int i = 0; i < steps; ++i) {
        if (sur_whole(s)) {
            NetArgs a = net_args(s, B);
            a.sample = 1;
            a.x = s.xbuf;
            a.ybuf = s.ybuf;
            a.count = s.count;
            a.have_host = have;
            a.cap = s.cap;
            a.seed = s.seed;
            a.step = s.sample_step++;
            a.recent = s.recent;
            const AdamStep step = adam_step(s);
            if ((e = whole_step(s, a, &step, s.loss, st))) return e;
            continue;
        }
        batch_kernel<<<(B * 32 + 255) / 256, 256, 0, st>>>(B, s.K, s.count, have, s.cap, s.seed, s.sample_step++,
                                                           s.recent, s.xbuf, s.ybuf, s.stats, s.xmin, s.xmax, s.tb,
                                                           s.Xb);
        if ((e = sur_backward(s, s.Xb, s.tb, B, s.loss, st))) return e;
        if ((e = sur_adam(s, st))) return e;
    }
    return cudaGetLastError();
}

cudaError_t sur_select(const float *key, int P, int k, int *rows, cudaStream_t st)
{
    select_kernel<<<1, 1024, 0, st>>>(key, P, k, rows);
    return cudaGetLastError();
}

cudaError_t sur_rank_corr(const double *fk, const int *rows, const float *logphi, int k, float *rho,
                          cudaStream_t st)
{
    rank_corr_kernel<<<1, 1024, 0, st>>>(fk, rows, logphi, k, rho);
    return cudaGetLastError();
}

cudaError_t sur_gather(const float *x, const int *rows, int k, int K, float *out, cudaStream_t st)
{
    gather_kernel<<<blocks_for((long long)k * K), 256, 0, st>>>(x, rows, k, K, out);
    return cudaGetLastError();
}

cudaError_t sur_scatter(const int *rows, const double *fk, int k, const float *logphi, int P,
                        double *fit, double *rank, cudaStream_t st)
{
    scatter_kernel<<<(P + 255) / 256, 256, 0, st>>>(rows, fk, k, logphi, P, fit, rank);
    scatter_fill_kernel<<<(k + 255) / 256, 256, 0, st>>>(rows, fk, k, fit, rank);
    return cudaGetLastError();
}

}  // namespace empso
