// Dense scan update: Eq. 9 on every state from a precomputed expected-range table.
//
// The map is static, so the expected range of every cell along A fixed directions 2 pi a / A
// (A a multiple of K, so bin k's heading is direction k A / K) is cast once with the FP32
// grid walk of the sampled update and stored as an 8-bit code [A][H][W]:
// q = floor(t * inv_step + 0.5) capped at 255, t in cells, each FP32 operation rounded.
// A scan then scores every state: beam b of bin k reads direction (k s + m_b) mod A, s = A/K,
// m_b its offset from the bin heading rounded to the table grid (host), and
//   log L(k, j, i) = -sum_b (z_b - q step)^2 / (2 sigma^2)
// over the used beams; then X <- X exp(log L - c) mult, c = max over states of
// (log L + log X): the most probable state after the update is stored at the storage
// multiplier, so an informative scan (Eq. 9's normaliser far below 1) cannot underflow FP16
// storage.  The new sum becomes the lazy normaliser (Eq. 9's eta).
//
// Kernels:
//  * range_table_kernel: one thread per cell walks all A directions; the writes of one
//    direction are consecutive across a warp.
//  * dense_score_kernel: a CTA of 256 threads stages the table columns of DC = 64 cells in shared
//    memory (16-byte loads), regrouped by residue r = a mod s with the K rows of each group twice,
//    so that no bin of a beam wraps.  A thread owns 4 cells and every 16th bin: one 4-byte load
//    gives the codes of 4 states, four byte permutes turn them into floats (the 2^23 exponent
//    trick, exact for 0 .. 255) and the terms run on the packed FP32 pipe, 2.9 instructions a
//    (state, beam) term.  A warp reads two rows of opposite parity: all 32 banks.  What bounds it:
//    instruction issue.  One thread per cell with 32 bins and a byte load per term took 4.5
//    instructions a term at 12 warps an SM, 373 us on 512 x 512 x 64 with 86 beams; this form
//    182 us.  It also reads the stored belief for the offset c.
//  * dense_apply_kernel: X exp(log L - c) mult stored with the storage type's rounding, FP32
//    Kahan partial sums per thread, FP64 per CTA, the last CTA combining them in a fixed
//    order.
#include <cfloat>
#include <climits>
#include <type_traits>

#include "dda.cuh"
#include "kernels.h"
#include "per_device.h"
#include "tiled_common.cuh"

namespace loc {
namespace {

constexpr int NT = 256;
constexpr int DC = 64;            // cells per score CTA
constexpr int SNT = 256;          // score threads: 16 quads of cells x 16 groups of bins
constexpr int NGRP = 16;

// Shared bytes of a score CTA's staged table: A / K residue blocks of 2 K rows of DC cells.
__host__ __device__ constexpr size_t dense_table_bytes(int A, int K) {
    (void)K;
    return 2 * (size_t)A * DC;
}

// Order-preserving map of floats to unsigned ints (for atomicMax on floats).
__device__ __forceinline__ unsigned int f2ord(float f) {
    const unsigned int u = __float_as_uint(f);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float ord2f(unsigned int u) {
    return __uint_as_float((u & 0x80000000u) ? (u & 0x7FFFFFFFu) : ~u);
}

__global__ void __launch_bounds__(NT) range_table_kernel(const uint8_t* __restrict__ trav, int H, int W,
                                                         const float* __restrict__ dirs, int A, float rmax,
                                                         float inv_step, uint8_t* __restrict__ out) {
    const size_t hw = (size_t)H * W;
    for (size_t c = (size_t)blockIdx.x * NT + threadIdx.x; c < hw; c += (size_t)gridDim.x * NT) {
        const int j = (int)(c / W), i = (int)(c % W);
        for (int a = 0; a < A; ++a) {
            const float t = dda_cells(trav, H, W, j, i, dirs[2 * a], dirs[2 * a + 1], rmax);
            const float f = floorf(__fadd_rn(__fmul_rn(t, inv_step), 0.5f));
            out[(size_t)a * hw + c] = (uint8_t)(f > 255.0f ? 255.0f : f);
        }
    }
}

// NB: bins per thread, bg, bg + 16, ...; FULL: K = 16 NB, so that their rows are constant offsets
// (else bins past K - 1 repeat the first one and are dropped).
template <typename T, int NB, bool FULL>
__global__ void __launch_bounds__(SNT) dense_score_kernel(const uint8_t* __restrict__ table,
                                                          const uint8_t* __restrict__ trav, const T* __restrict__ B,
                                                          size_t hw, int K, int A, int s, const int* __restrict__ m,
                                                          const float* __restrict__ zs, int nu, float scale,
                                                          float* __restrict__ logL, unsigned int* maxL) {
    // Us[(r 2K + k') DC + t] = code of direction ((k' mod K) s + r) for cell c0 + t, k' < 2K: bins
    // 0 .. K - 1 of a beam with m = q s + r sit at rows r 2K + q + 0 .. K - 1.
    extern __shared__ __align__(16) unsigned char dsm[];
    using tiled::f2;
    uint8_t* Us = dsm;
    int2* sm_b = reinterpret_cast<int2*>(dsm + dense_table_bytes(A, K));  // [nu] byte offset of a beam's first row; its z
    const int t = threadIdx.x;
    const size_t c0 = (size_t)blockIdx.x * DC;
    auto put = [&](int a, auto store) {                           // direction a's two rows
        const int r = a % s, k = a / s;
        store(r * 2 * K + k);
        store(r * 2 * K + K + k);
    };
    if ((hw & 15) == 0 && c0 + DC <= hw) {
        // 16 cells per 16-byte load: DC / 16 threads per direction, four passes in flight
        constexpr int TPD = DC / 16;
        const int g = t % TPD, a0 = t / TPD;
#pragma unroll 4
        for (int a = a0; a < A; a += SNT / TPD) {
            const uint4 v = *reinterpret_cast<const uint4*>(table + (size_t)a * hw + c0 + 16 * g);
            put(a, [&](int row) { *reinterpret_cast<uint4*>(Us + (size_t)row * DC + 16 * g) = v; });
        }
    } else {
        for (int q = t; q < A * DC; q += SNT) {
            const int a = q / DC, i = q % DC;
            const uint8_t v = c0 + i < hw ? table[(size_t)a * hw + c0 + i] : (uint8_t)0;
            put(a, [&](int row) { Us[(size_t)row * DC + i] = v; });
        }
    }
    for (int u = t; u < nu; u += SNT) {
        sm_b[u] = make_int2(((m[u] % s) * 2 * K + m[u] / s) * DC, __float_as_int(zs[u]));
    }
    __syncthreads();
    const int quad = t & 15, bg = t >> 4;
    const uint8_t* mine[FULL ? 1 : NB];                           // the thread's bins, from a beam's first row
#pragma unroll
    for (int n = 0; n < (FULL ? 1 : NB); ++n) mine[n] = Us + (bg + NGRP * n < K ? bg + NGRP * n : 0) * DC + 4 * quad;
    f2 acc[NB][2];
#pragma unroll
    for (int n = 0; n < NB; ++n) acc[n][0] = acc[n][1] = 0ull;
    const f2 bias = tiled::pk(-8388608.0f, -8388608.0f);
    // each lane of a pair is one state: the beams in order, the same sums bit for bit whichever
    // thread takes it
#pragma unroll 2
    for (int u = 0; u < nu; ++u) {
        const int2 b = sm_b[u];
        const f2 zu = tiled::pk(__int_as_float(b.y), __int_as_float(b.y));
#pragma unroll
        for (int n = 0; n < NB; ++n) {
            const uint32_t q = *reinterpret_cast<const uint32_t*>((FULL ? mine[0] + n * NGRP * DC : mine[FULL ? 0 : n]) + b.x);
            // the codes as floats (2^23 + q, exact, minus 2^23)
            const f2 q0 = tiled::fadd2(tiled::pk(__uint_as_float(__byte_perm(q, 0x4B000000u, 0x7650)),
                                                 __uint_as_float(__byte_perm(q, 0x4B000000u, 0x7651))), bias);
            const f2 q1 = tiled::fadd2(tiled::pk(__uint_as_float(__byte_perm(q, 0x4B000000u, 0x7652)),
                                                 __uint_as_float(__byte_perm(q, 0x4B000000u, 0x7653))), bias);
            const f2 d0 = tiled::fsub2(zu, q0), d1 = tiled::fsub2(zu, q1);
            acc[n][0] = tiled::ffma2(d0, d0, acc[n][0]);
            acc[n][1] = tiled::ffma2(d1, d1, acc[n][1]);
        }
    }
    const size_t c = c0 + 4 * quad;
    bool free[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) free[e] = c + e < hw && trav[c + e] != 0;
    const bool whole = (hw & 3) == 0 && c + 4 <= hw;              // 16-byte rows of four cells
    float best = -FLT_MAX;
#pragma unroll
    for (int n = 0; n < NB; ++n) {
        const int k = bg + NGRP * n;
        if (k >= K) break;
        float a[4], l[4];
        tiled::upk(acc[n][0], a[0], a[1]);
        tiled::upk(acc[n][1], a[2], a[3]);
        const size_t q = (size_t)k * hw + c;
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            l[e] = free[e] ? -a[e] * scale : -INFINITY;
            const float x = c + e < hw ? Store<T>::ld(B + q + e) : 0.0f;
            if (free[e] && x > 0.0f) best = fmaxf(best, l[e] + logf(x));
        }
        if (whole) {
            *reinterpret_cast<float4*>(logL + q) = make_float4(l[0], l[1], l[2], l[3]);
        } else {
            for (int e = 0; e < 4; ++e)
                if (c + e < hw) logL[q + e] = l[e];
        }
    }
    for (int o = 16; o > 0; o >>= 1) best = fmaxf(best, __shfl_down_sync(0xffffffffu, best, o));
    if ((t & 31) == 0 && best > -FLT_MAX) atomicMax(maxL, f2ord(best));
}

// V neighbouring cells per thread (one for FP32, a 4-byte pair for 16-bit storage), their bins in
// order: the BF16 rounding residual of a cell runs along theta.  What bounds it: the two reads and
// the write of every state, so four bins' loads are in flight per thread (51 us at 512 x 512 x 64
// FP32 with one, 44 with four; four cells a thread left too few warps, 60).
template <typename T, int V> struct Cells;
template <> struct Cells<float, 2> {
    static __device__ __forceinline__ void ld(const float* p, float (&v)[2]) {
        const float2 a = *reinterpret_cast<const float2*>(p);
        v[0] = a.x; v[1] = a.y;
    }
};
template <typename T> struct Cells<T, 2> {                        // 16-bit
    static __device__ __forceinline__ void ld(const T* p, float (&v)[2]) {
        union {
            uint32_t u;
            T x[2];
        } raw;
        raw.u = *reinterpret_cast<const uint32_t*>(p);
#pragma unroll
        for (int e = 0; e < 2; ++e) v[e] = Store<T>::ld(&raw.x[e]);
    }
};
template <typename T> struct Cells<T, 1> {
    static __device__ __forceinline__ void ld(const T* p, float (&v)[1]) { v[0] = Store<T>::ld(p); }
};

template <typename T, int V>
__global__ void __launch_bounds__(NT) dense_apply_kernel(T* __restrict__ B, const float* __restrict__ logL, size_t hw,
                                                         int K, const unsigned int* maxL, float log_mult,
                                                         double* partials, SessionDev* sd) {
    __shared__ double red[NT / 32];
    const float c = ord2f(*maxL);                 // max of log L + log X
    const float off = log_mult - c;
    KahanF acc;
    for (size_t cell = V * ((size_t)blockIdx.x * NT + threadIdx.x); cell < hw; cell += V * (size_t)gridDim.x * NT) {
        float res[V];
#pragma unroll
        for (int e = 0; e < V; ++e) res[e] = 0.0f;
        for (int k0 = 0; k0 < K; k0 += 4) {
            float x[4][V], l[4][V];
#pragma unroll
            for (int d = 0; d < 4; ++d)
                if (k0 + d < K) {
                    Cells<T, V>::ld(B + (size_t)(k0 + d) * hw + cell, x[d]);
                    Cells<float, V>::ld(logL + (size_t)(k0 + d) * hw + cell, l[d]);
                }
#pragma unroll
            for (int d = 0; d < 4; ++d) {
                if (k0 + d >= K) break;
                struct alignas(V * sizeof(T)) Out {
                    T y[V];
                } o;
#pragma unroll
                for (int e = 0; e < V; ++e) {
                    // x exp(log L + off) <= mult; for a small x the factor alone could overflow, so a
                    // large exponent takes log x in (the multiply keeps x's precision elsewhere)
                    const float z = l[d][e] + off, xe = x[d][e];
                    const float v = xe > 0.0f ? (z < 80.0f ? xe * expf(z) : expf(z + logf(xe))) : 0.0f;
                    acc.add(store_diffused<T>(&o.y[e], v, res[e]));
                }
                *reinterpret_cast<Out*>(B + (size_t)(k0 + d) * hw + cell) = o;
            }
        }
    }
    const double bt = block_sum<NT>(acc.value(), red);
    const unsigned int nblocks = gridDim.x;
    finish_sum<NT>(bt, partials, &sd->counter, nblocks, red, [sd, c, log_mult](double S) {
        const double Z0 = sd->Z;
        if (S > 0.0 && isfinite(S)) {
            // Eq. 9's normaliser: sum(b exp(log L)) = S exp(c) / (mult Z0)
            sd->Z = S;
            sd->inv_Z = (float)(1.0 / S);
            sd->logscale += log(S) - log(Z0) + (double)c - (double)log_mult;
        } else {
            if (!isfinite(S)) sd->status |= LOC_DEV_ERR_NONFINITE_Z;
            sd->Z = 1.0;
            sd->inv_Z = 1.0f;
            sd->reinit = 1;
            sd->n_reinit += 1;
        }
    });
}

// Probe columns for the map difficulty: out[p A + a] = table[a][probes[p]], flag[p] = M there.
__global__ void __launch_bounds__(NT) gather_columns_kernel(const uint8_t* __restrict__ table,
                                                            const uint8_t* __restrict__ trav, size_t hw, int A,
                                                            const int32_t* __restrict__ probes, int n,
                                                            uint8_t* __restrict__ out, uint8_t* __restrict__ flag) {
    const size_t total = (size_t)n * A;
    for (size_t q = (size_t)blockIdx.x * NT + threadIdx.x; q < total; q += (size_t)gridDim.x * NT) {
        const int p = (int)(q / A), a = (int)(q % A);
        out[q] = table[(size_t)a * hw + probes[p]];
        if (a == 0) flag[p] = trav[probes[p]];
    }
}

__device__ __forceinline__ bool better_f(float v, long long i, float bv, long long bi) {
    return v > bv || (v == bv && i < bi);
}

// argmax of a float array (the first index among equal values): per-thread scans in
// increasing index order, warps and CTAs combined with better_f, the last CTA combining the
// CTA results in a fixed order and writing the index to *out.
__global__ void __launch_bounds__(NT) argmax_f32_kernel(const float* __restrict__ x, size_t n, float* pv,
                                                        long long* pi, unsigned int* counter, long long* out) {
    __shared__ float sv[NT / 32];
    __shared__ long long si[NT / 32];
    __shared__ int s_last;
    float bv = -INFINITY;
    long long bi = LLONG_MAX;
    for (size_t q = (size_t)blockIdx.x * NT + threadIdx.x; q < n; q += (size_t)gridDim.x * NT) {
        const float v = x[q];
        if (better_f(v, (long long)q, bv, bi)) {
            bv = v;
            bi = (long long)q;
        }
    }
    auto reduce = [&]() {
        for (int o = 16; o > 0; o >>= 1) {
            const float ov = __shfl_down_sync(0xffffffffu, bv, o);
            const long long oi = __shfl_down_sync(0xffffffffu, bi, o);
            if (better_f(ov, oi, bv, bi)) {
                bv = ov;
                bi = oi;
            }
        }
        const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
        __syncthreads();
        if (lane == 0) {
            sv[warp] = bv;
            si[warp] = bi;
        }
        __syncthreads();
        if (threadIdx.x == 0)
            for (int w = 1; w < NT / 32; ++w)
                if (better_f(sv[w], si[w], bv, bi)) {
                    bv = sv[w];
                    bi = si[w];
                }
    };
    reduce();
    if (threadIdx.x == 0) {
        pv[blockIdx.x] = bv;
        pi[blockIdx.x] = bi;
        __threadfence();
        s_last = atomicAdd(counter, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    bv = -INFINITY;
    bi = LLONG_MAX;
    for (unsigned int b = threadIdx.x; b < gridDim.x; b += NT) {
        const float v = ((volatile float*)pv)[b];
        const long long q = ((volatile long long*)pi)[b];
        if (better_f(v, q, bv, bi)) {
            bv = v;
            bi = q;
        }
    }
    reduce();
    if (threadIdx.x == 0) {
        *out = bi;
        *counter = 0u;
    }
}

}  // namespace

constexpr unsigned int kArgmaxF32Blocks = 512;

size_t argmax_f32_scratch_bytes() { return (size_t)kArgmaxF32Blocks * (sizeof(float) + sizeof(long long)) + 16; }

cudaError_t launch_gather_columns(const uint8_t* table, const uint8_t* trav, int H, int W, int A,
                                  const int32_t* probes, int n, uint8_t* out, uint8_t* flag, cudaStream_t st) {
    const size_t total = (size_t)n * A;
    size_t nb = (total + NT - 1) / NT;
    if (nb > 4096) nb = 4096;
    if (nb < 1) nb = 1;
    gather_columns_kernel<<<(unsigned int)nb, NT, 0, st>>>(table, trav, (size_t)H * W, A, probes, n, out, flag);
    return cudaGetLastError();
}

cudaError_t launch_argmax_f32(const float* x, size_t n, void* scratch, long long* out, cudaStream_t st) {
    long long* pi = (long long*)scratch;
    float* pv = (float*)(pi + kArgmaxF32Blocks);
    unsigned int* counter = reinterpret_cast<unsigned int*>(pv + kArgmaxF32Blocks);
    size_t nb = (n + NT - 1) / NT;
    if (nb > kArgmaxF32Blocks) nb = kArgmaxF32Blocks;
    if (nb < 1) nb = 1;
    argmax_f32_kernel<<<(unsigned int)nb, NT, 0, st>>>(x, n, pv, pi, counter, out);
    return cudaGetLastError();
}

size_t dense_score_smem(int A, int K, int nu) { return dense_table_bytes(A, K) + (size_t)nu * 8; }

cudaError_t launch_range_table(const uint8_t* trav, int H, int W, const float* dirs, int A, float rmax,
                               float inv_step, uint8_t* out, cudaStream_t st) {
    const size_t hw = (size_t)H * W;
    size_t nb = (hw + NT - 1) / NT;
    if (nb > 65535) nb = 65535;
    range_table_kernel<<<(unsigned int)nb, NT, 0, st>>>(trav, H, W, dirs, A, rmax, inv_step, out);
    return cudaGetLastError();
}

template <typename T, int NB, bool FULL>
cudaError_t score_nb(const uint8_t* table, const uint8_t* trav, const void* B, size_t hw, int K, int A, const int* m,
                     const float* zs, int nu, float scale, float* logL, unsigned int* maxL, cudaStream_t st) {
    const size_t smem = dense_score_smem(A, K, nu);
    // one size for every launch: with the launch's own, a thread with a small table could lower the limit
    // between another's setting it and its launch
    static PerDevice ready;
    int dev = 0, set = 0;
    cudaGetDevice(&dev);
    const cudaError_t e = ready.get(dev, &set, [](int* n) {
        *n = 1;
        return cudaFuncSetAttribute(dense_score_kernel<T, NB, FULL>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)dense_score_smem(LOC_MAX_TABLE_DIRS, 1, LOC_MAX_DENSE_BEAMS));
    });
    if (e != cudaSuccess) return e;
    const unsigned int nb = (unsigned int)((hw + DC - 1) / DC);
    dense_score_kernel<T, NB, FULL><<<nb, SNT, smem, st>>>(table, trav, static_cast<const T*>(B), hw, K, A, A / K, m, zs, nu,
                                                     scale, logL, maxL);
    return cudaGetLastError();
}

template <typename T>
cudaError_t score_t(const uint8_t* table, const uint8_t* trav, const void* B, int H, int W, int K, int A,
                    const int* m, const float* zs, int nu, float scale, float* logL, unsigned int* maxL,
                    cudaStream_t st) {
    const size_t hw = (size_t)H * W;
#define LOC_NB(N)                                                                                        \
    return K == NGRP * N ? score_nb<T, N, true>(table, trav, B, hw, K, A, m, zs, nu, scale, logL, maxL, st) \
                         : score_nb<T, N, false>(table, trav, B, hw, K, A, m, zs, nu, scale, logL, maxL, st)
    switch ((K + NGRP - 1) / NGRP) {               // bins per thread (LOC_MAX_K = 256: 16 at most)
        case 1: LOC_NB(1);
        case 2: LOC_NB(2);
        case 3: LOC_NB(3);
        case 4: LOC_NB(4);
        case 5: LOC_NB(5);
        case 6: LOC_NB(6);
        case 7: case 8: LOC_NB(8);
        default: LOC_NB(16);
    }
#undef LOC_NB
}

cudaError_t launch_dense_score(const uint8_t* table, const uint8_t* trav, const void* B, int storage, int H, int W,
                               int K, int A, const int* m, const float* zs, int nu, float scale, float* logL,
                               unsigned int* maxL, cudaStream_t st) {
    if (A % K != 0) return cudaErrorInvalidValue;
    switch (storage) {
        case LOC_F32: return score_t<float>(table, trav, B, H, W, K, A, m, zs, nu, scale, logL, maxL, st);
        case LOC_BF16: return score_t<__nv_bfloat16>(table, trav, B, H, W, K, A, m, zs, nu, scale, logL, maxL, st);
        case LOC_F16: return score_t<__half>(table, trav, B, H, W, K, A, m, zs, nu, scale, logL, maxL, st);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_dense_apply(void* B, int storage, const float* logL, size_t hw, int K, const unsigned int* maxL,
                               float log_mult, double* partials, unsigned int nparts, SessionDev* sd,
                               cudaStream_t st) {
    const int v = storage != LOC_F32 && hw % 2 == 0 ? 2 : 1;
    size_t nb = (hw / v + NT - 1) / NT;
    if (nb > nparts) nb = nparts;
    if (nb > 4096) nb = 4096;
    if (nb < 1) nb = 1;
    const unsigned int n = (unsigned int)nb;
#define LOC_APPLY(T)                                                                                            \
    if (v == 2) dense_apply_kernel<T, 2><<<n, NT, 0, st>>>((T*)B, logL, hw, K, maxL, log_mult, partials, sd);      \
    else dense_apply_kernel<T, 1><<<n, NT, 0, st>>>((T*)B, logL, hw, K, maxL, log_mult, partials, sd)
    switch (storage) {
        case LOC_F32: dense_apply_kernel<float, 1><<<n, NT, 0, st>>>((float*)B, logL, hw, K, maxL, log_mult, partials, sd); break;
        case LOC_BF16: LOC_APPLY(__nv_bfloat16); break;
        case LOC_F16: LOC_APPLY(__half); break;
        default: return cudaErrorInvalidValue;
    }
#undef LOC_APPLY
    return cudaGetLastError();
}

}  // namespace loc
