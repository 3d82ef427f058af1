// LIDAR sample update of Section III-B: belief map -> Floyd-Steinberg sample selection
// (III-B.1) -> expected ranges by grid ray casting -> Gaussian range likelihood -> Eq. 9 on
// the sampled states (the sampled set keeps its mass).
//
// The two steps whose results are integers decided by floating point -- the dithering and
// the ray walk -- use FP32 with every operation explicitly rounded (__fadd_rn / __fmul_rn /
// __fdiv_rn, so nothing is contracted into an FMA) in a fixed order.
#include <algorithm>
#include <cfloat>

#include <cooperative_groups.h>
#include <type_traits>

#include "dda.cuh"
#include "kernels.h"
#include "per_device.h"

namespace loc {
namespace {

constexpr int NT = 256;
constexpr unsigned long long kSpinNs = 200ull * 1000 * 1000;

// Limit of the bounded waits of the Floyd-Steinberg block hand-offs, and the test hook that
// makes them wait on a flag nothing sets (so that the limit runs out and the kernel returns
// with LOC_DEV_ERR_TIMEOUT).  Set by set_fs_wait (loc_debug_fs_stall).
__device__ unsigned long long g_fs_wait_ns = kSpinNs;
__device__ int g_fs_stall = 0;

__device__ __forceinline__ unsigned long long gtime() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// ------------------------------------------------------------------ belief map and fs

// m[q] = max_k belief(k, q) (normalised, FP32); the last CTA writes fs = n_samples / sum(m)
// (FP64 sum, rounded to FP32), or 0 when the map is empty.
template <typename T>
__global__ void __launch_bounds__(NT) belief_map_kernel(const T* __restrict__ B, const uint8_t* __restrict__ trav,
                                                        SessionDev* sd, float inv_uniform, size_t hw, int K,
                                                        float* __restrict__ m, double* partials,
                                                        unsigned int* counter, int n_samples, float* fs_out) {
    __shared__ double red[NT / 32];
    const int reinit = sd->reinit;
    const float scale = sd->inv_Z;
    KahanF acc;
    for (size_t q = (size_t)blockIdx.x * NT + threadIdx.x; q < hw; q += (size_t)gridDim.x * NT) {
        float v = 0.0f;
        if (reinit) {
            v = (float)trav[q] * inv_uniform;
        } else {
            for (int k = 0; k < K; ++k) v = fmaxf(v, Store<T>::ld(B + (size_t)k * hw + q) * scale);
        }
        m[q] = v;
        acc.add(v);
    }
    const double bt = block_sum<NT>(acc.value(), red);
    finish_sum<NT>(bt, partials, counter, gridDim.x, red, [fs_out, n_samples](double S) {
        *fs_out = S > 0.0 ? (float)((double)n_samples / S) : 0.0f;
    });
}

// The same with V consecutive cells per thread and 16-byte loads (hw a multiple of V).
template <typename T, int V>
__global__ void __launch_bounds__(NT) belief_map_vec_kernel(const T* __restrict__ B, const uint8_t* __restrict__ trav,
                                                            SessionDev* sd, float inv_uniform, size_t hw, int K,
                                                            float* __restrict__ m, double* partials,
                                                            unsigned int* counter, int n_samples, float* fs_out) {
    static_assert(V * sizeof(T) == 16, "one 16-byte load per plane");
    __shared__ double red[NT / 32];
    const int reinit = sd->reinit;
    const float scale = sd->inv_Z;
    KahanF acc;
    const size_t ng = hw / V;
    for (size_t g = (size_t)blockIdx.x * NT + threadIdx.x; g < ng; g += (size_t)gridDim.x * NT) {
        float v[V];
#pragma unroll
        for (int e = 0; e < V; ++e) v[e] = 0.0f;
        if (reinit) {
#pragma unroll
            for (int e = 0; e < V; ++e) v[e] = (float)trav[g * V + e] * inv_uniform;
        } else {
#pragma unroll 8
            for (int k = 0; k < K; ++k) {                      // eight planes' loads in flight
                union {
                    uint4 u;
                    T x[V];
                } raw;
                raw.u = __ldg(reinterpret_cast<const uint4*>(B + (size_t)k * hw) + g);
#pragma unroll
                for (int e = 0; e < V; ++e) v[e] = fmaxf(v[e], Store<T>::ld(&raw.x[e]) * scale);
            }
        }
#pragma unroll
        for (int e = 0; e < V; e += 4)
            *reinterpret_cast<float4*>(m + g * V + e) = make_float4(v[e], v[e + 1], v[e + 2], v[e + 3]);
#pragma unroll
        for (int e = 0; e < V; ++e) acc.add(v[e]);
    }
    const double bt = block_sum<NT>(acc.value(), red);
    finish_sum<NT>(bt, partials, counter, gridDim.x, red, [fs_out, n_samples](double S) {
        *fs_out = S > 0.0 ? (float)((double)n_samples / S) : 0.0f;
    });
}

// ------------------------------------------------------------------ Floyd-Steinberg

// Warp w of a cluster of kFsWarps-warp CTAs takes the 32-row blocks w, w + (all warps), ...; lane l
// owns row 32 rb + l and handles column i = t - 3 l at step t.  The three errors it needs from the
// row above (columns i - 1, i, i + 1) were produced by lane l - 1 at steps t - 4, t - 3 and t - 2
// and arrive by warp shuffle one step before they are used, so only the lane's own error chain
// (multiply, two adds, compare) is left between two steps.
//
// What bounds it: the chain.  A row can take column i only when the row above has taken i + 1, so
// the whole map is a wavefront of W + 94 + (blocks - 1) x (94 + hand-off) steps.  One CTA of 16
// warps (four rows of blocks one after the other, 16 warps on four schedulers, a fence per
// hand-off) took 1.73 ms at 2048 x 2048; a warp per block on a scheduler of its own, with
// hand-offs that need no fence, takes 0.40 (60-odd cycles a step, ten thousand cycles from a block's
// start to the next one's).  The cluster keeps the warps that wait on one another resident together.
//
// Hand-off: a block's last lane writes its errors into the next block's inbox as it goes: shared
// memory of the next block's CTA, through the cluster (bnd in global memory where the rows are too
// long for that: ~1000 cycles a hand-off, 0.82 ms at 2048 x 2048).  An inbox starts as kFsEmpty (a
// NaN that no arithmetic produces), so a value that is not kFsEmpty is there and needs no fence: the
// next block polls the kFsSub values it needs next, with a limit.
//
// A second warp per block brings the map: a ring of six 32-column chunks per row in shared memory
// (column i at position i mod 192), the first chunk repeated behind the sixth so that a window of
// 32 steps reads at constant offsets; a pitch of 226 makes the lanes' 3-column skew hit distinct
// banks.  A window reads chunks T - 3 .. T, so the ring is two chunks ahead.  (Done by the block's
// own warp between its windows, the copy took a third of the time.)  Selections are bits: a lane collects a window's
// 32 and writes them as one aligned word of its row.  Terms of the error sum whose source lies
// outside the grid are zero (their errors were never produced), so the sum always takes the same
// four terms in the same order; only the right neighbour above is masked at the last column.
constexpr size_t kScoreWindowBytes = 96 * 1024;   // shared memory for the score kernel's map window
constexpr int kScoreNT = 384;                      // score kernel threads: 360 beam directions in one round
constexpr int kFsWarps = 4;               // one per scheduler
constexpr int kFsMaxCtas = 16;            // largest cluster: 64 blocks of 32 rows side by side
constexpr int kFsSkew = 3;
constexpr int kFsLead = 32 * kFsSkew;     // steps of skew over a block, rounded up: 93 -> 96
constexpr int kFsChunks = 6, kFsRing = 32 * kFsChunks, kFsPitch = 226;
constexpr uint32_t kFsEmpty = 0xFFFFFFFFu;
constexpr int kFsSub = 16;                // steps between two looks at the inbox
constexpr int kFsPad = kFsSub - 1;        // column c of an inbox lies at c + 15: looks are aligned
constexpr size_t kFsRingBytes = sizeof(float) * kFsWarps * 32 * kFsPitch;
constexpr size_t kFsInboxBytes = 108 * 1024;   // shared memory for the inboxes of a CTA at most

// inboxes a warp: two where it takes several blocks (the block above its next one may write while
// it still reads), each W rounded up to a multiple of 32
template <bool DSM>
__global__ void __launch_bounds__(kFsWarps * 64) fs_kernel(const float* __restrict__ m, const float* fs_ptr, int H,
                                                           int W, uint32_t* __restrict__ selbits,
                                                           int* __restrict__ rowcnt, float* bnd, int nbox, int* status) {
    extern __shared__ __align__(16) float fs_ring_all[];
    __shared__ volatile int s_filled[kFsWarps], s_done[kFsWarps];   // chunks brought, windows done
    namespace cg = cooperative_groups;
    const int lane = threadIdx.x & 31, warp = (threadIdx.x >> 5) % kFsWarps;
    const bool loader = threadIdx.x >= kFsWarps * 32;
    float* ring = fs_ring_all + (size_t)warp * 32 * kFsPitch;
    const unsigned long long wait_ns = g_fs_wait_ns;
    const int stall = g_fs_stall;
    const int nrb = (H + 31) / 32, nch = (W + 31) / 32;
    const int nwin = (W + kFsSkew * 31 + 31) / 32;
    const float w7 = 0.4375f, w3 = 0.1875f, w5 = 0.3125f, w1 = 0.0625f;
    const int wpad = 32 * nch + 64;
    float* box_all = fs_ring_all + kFsRingBytes / sizeof(float);
    auto inbox = [&](int w, int round) { return box_all + (size_t)(w * nbox + (nbox == 2 ? round & 1 : 0)) * wpad; };
    if (threadIdx.x < kFsWarps) s_filled[threadIdx.x] = s_done[threadIdx.x] = 0;
    if constexpr (DSM) {
        for (int q = threadIdx.x; q < kFsWarps * nbox * wpad; q += kFsWarps * 64) box_all[q] = __uint_as_float(kFsEmpty);
        cg::this_cluster().sync();
    } else {
        __syncthreads();
    }
    bool failed = false;
    // a whole warp's wait with a limit; ready() gives every lane the same answer
    auto await = [&](auto ready) {
        if (ready()) return;
        const unsigned long long g0 = gtime();
        for (unsigned int it = 0; !ready();) {
            if (loader) __nanosleep(200);                      // two chunks ahead: leave the pipes to the steps
            if (__any_sync(0xffffffffu, ++it > (1u << 24) || gtime() - g0 > wait_ns)) {
                if (lane == 0) atomicOr(status, LOC_DEV_ERR_TIMEOUT);
                failed = true;                                 // the blocks below run into their limits too
                return;
            }
        }
    };
    int round = 0;
    for (int rb = blockIdx.x * kFsWarps + warp; rb < nrb && !failed; rb += gridDim.x * kFsWarps, ++round) {
        const int j0 = 32 * rb, j = j0 + lane;
        const bool row_ok = j < H;
        const bool interior = j0 + 31 < H;                     // every row of the block in the grid
        if (loader) {
            const float fs = *fs_ptr;
            float pre[32];                                     // column 32 c + lane of rows j0 ..
            auto load_chunk = [&](int c) {
                const int col = 32 * c + lane;
                const float* src = m + (size_t)j0 * W + col;
#pragma unroll
                for (int r = 0; r < 32; ++r) pre[r] = (interior || j0 + r < H) && col < W ? __ldg(src + (size_t)r * W) : 0.0f;
            };
            load_chunk(0);
            for (int c = 0; c < nch && !failed; ++c) {
                // chunk c takes the place of chunk c - 6, last read in window c - 3; the first chunk
                // waits for the end of the block before
                const int need = round * nwin + (c >= kFsChunks - 3 ? c - (kFsChunks - 4) : 0);
                await([&]() { return s_done[warp] >= need; });
                __syncwarp();
                float* dst = ring + (c % kFsChunks) * 32 + lane;
#pragma unroll
                for (int r = 0; r < 32; ++r) {
                    float v = __fmul_rn(pre[r], fs);
                    if (v > 1.0f) v = 1.0f;
                    dst[r * kFsPitch] = v;
                    if (c % kFsChunks == 0) dst[r * kFsPitch + kFsRing] = v;
                }
                __threadfence_block();
                __syncwarp();
                if (lane == 0) s_filled[warp] = round * nch + c + 1;
                if (c + 1 < nch) load_chunk(c + 1);
            }
            continue;
        }
        const float* own = ring + lane * kFsPitch;             // this lane's row
        float up_old = 0.0f, up_mid = 0.0f, up_new = 0.0f;   // row above: columns i-1, i, i+1
        float pend = 0.0f;                                     // ... and the next one, for the next step
        float last = 0.0f;                                     // own error at the column before
        uint32_t before = 0;                                   // the previous window's selections
        int cnt = 0;
        const int r_off = (kFsLead - kFsSkew * lane) & 31;     // (t0 - 3 lane) mod 32, t0 a multiple of 32
        const bool publish = lane == 31 && rb + 1 < nrb;       // the next block reads this row
        float* below;                                          // the next block's inbox, and this one's
        const volatile uint32_t* above;
        if constexpr (DSM) {
            const int cta = blockIdx.x + (warp + 1) / kFsWarps, to = cta % gridDim.x;
            below = cg::this_cluster().map_shared_rank(inbox((warp + 1) % kFsWarps, round + cta / gridDim.x), to) + kFsPad;
            above = reinterpret_cast<const volatile uint32_t*>(inbox(warp, round) + kFsPad);
        } else {
            below = bnd + (size_t)(rb + 1 < nrb ? rb + 1 : rb) * W;
            above = reinterpret_cast<const volatile uint32_t*>(bnd) + (size_t)rb * W;
        }
        // the row above at columns c0 .. c0 + 15, c0 = 1 mod 16 (0 past the last one), every lane the same
        struct Above {
            uint32_t v[kFsSub];
        };
        auto look = [&](int c0) {
            Above e;
#pragma unroll
            for (int k = 0; k < kFsSub; ++k) e.v[k] = 0u;
            if (rb > 0 && c0 < W) {                            // (an inbox is padded past its last column)
                if constexpr (DSM) {
#pragma unroll
                    for (int h = 0; h < kFsSub / 4; ++h) {
                        uint32_t* v = e.v + 4 * h;
                        asm volatile("ld.volatile.shared.v4.u32 {%0, %1, %2, %3}, [%4];"
                                     : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3])
                                     : "r"((uint32_t)__cvta_generic_to_shared(const_cast<uint32_t*>(above) + c0 + 4 * h)));
                    }
#pragma unroll
                    for (int k = 0; k < kFsSub; ++k)
                        if (c0 + k >= W) e.v[k] = 0u;
                } else {
#pragma unroll
                    for (int k = 0; k < kFsSub; ++k)
                        if (c0 + k < W) e.v[k] = above[c0 + k];
                }
            }
            return e;
        };
        auto there = [&](const Above& e) {
            uint32_t most = 0;                                 // kFsEmpty is the largest word
#pragma unroll
            for (int k = 0; k < kFsSub; ++k) most = max(most, e.v[k]);
            return __all_sync(0xffffffffu, most != kFsEmpty && !(stall && rb > 0)) != 0;
        };
        // lane 0 starts at column 0 at once: the row above at column 0 must already be in its register
        // chain (other lanes shift theirs in while they wait to start)
        if (rb > 0) {
            uint32_t v = kFsEmpty;
            await([&]() {
                v = above[0];
                return __all_sync(0xffffffffu, !stall && v != kFsEmpty) != 0;
            });
            if (lane == 0) up_new = __uint_as_float(v);
        }
        Above next = look(1);
        int at = (kFsRing - kFsSkew * lane) % kFsRing;         // ring position of the lane's column at t0
        for (int T = 0; T < nwin && !failed; ++T) {
            const int t0 = 32 * T, have = round * nch + (T < nch ? T : nch - 1);
            await([&]() { return s_filled[warp] > have; });
            __syncwarp();
            const float* ow = own + at;
            uint32_t bits = 0;
            const bool plain = interior && t0 >= kFsSkew * 31 && t0 + 31 <= W - 2;
#pragma unroll
            for (int u = 0; u < 32; u += kFsSub) {
                Above now = next;
                if (!there(now)) await([&]() {
                    now = look(t0 + u + 1);
                    return there(now);
                });
                if (failed) break;
                next = look(t0 + u + 1 + kFsSub);
                float v[kFsSub];
#pragma unroll
                for (int k = 0; k < kFsSub; ++k) v[k] = ow[u + k];
                // In a plain window every lane's column lies in [0, W - 2] and every row of the block is in
                // the grid: no guards.  The others keep a lane's error as it is while its column is off the
                // grid (0 before the first one) and mask the right neighbour above at the last column; the
                // same operations in the same order (0 + x == x exactly).
                auto steps = [&](auto guarded) {
                    constexpr bool G = decltype(guarded)::value;
#pragma unroll
                    for (int k = 0; k < kFsSub; ++k) {
                        const int i = t0 + u + k - kFsSkew * lane;
                        up_old = up_mid;
                        up_mid = up_new;
                        up_new = lane == 0 ? __uint_as_float(now.v[k]) : pend;
                        pend = __shfl_up_sync(0xffffffffu, last, 1);
                        const bool in = !G || (row_ok && (unsigned)i < (unsigned)W);
                        float E = __fmul_rn(up_old, w1);
                        E = __fadd_rn(E, __fmul_rn(up_mid, w5));
                        E = __fadd_rn(E, __fmul_rn(G && i + 1 >= W ? 0.0f : up_new, w3));
                        E = __fadd_rn(E, __fmul_rn(last, w7));
                        const float val = __fadd_rn(v[k], E), less = __fsub_rn(val, 1.0f);
                        const bool on = val >= 0.5f;
                        const float err = on ? less : val;
                        last = in ? err : last;
                        bits |= on && in ? 1u << (u + k) : 0u;
                        if (publish && in) *reinterpret_cast<volatile float*>(below + i) = err;
                    }
                };
                if (plain) steps(std::false_type{});
                else steps(std::true_type{});
            }
            if (failed) break;
            __syncwarp();
            if (lane == 0) s_done[warp] = round * nwin + T + 1;
            at += 32;
            if (at >= kFsRing) at -= kFsRing;
            // the aligned word that this window completes: columns t0 - 3 lane - r_off ..
            const int c = (t0 - kFsSkew * lane - r_off) >> 5;
            const uint32_t word = __funnelshift_l(before, bits, r_off);
            before = bits;
            if (row_ok && c >= 0 && c < nch) {
                selbits[(size_t)j * nch + c] = word;
                cnt += __popc(word);
            }
        }
        if (failed) break;
        // the word that a lane's last window began, where it lies in the grid
        const int c = (32 * nwin - kFsSkew * lane - r_off) >> 5;
        if (row_ok && r_off > 0 && c >= 0 && c < nch) {
            const uint32_t word = before >> (32 - r_off);
            selbits[(size_t)j * nch + c] = word;
            cnt += __popc(word);
        }
        if (row_ok) rowcnt[j] = cnt;
        if constexpr (DSM) {                                   // empty again for the block after next
            if (nbox == 2) {
                float* box = inbox(warp, round);
                for (int q = lane; q < wpad; q += 32) box[q] = __uint_as_float(kFsEmpty);
                __threadfence();
                __syncwarp();
            }
        }
    }
    // no CTA leaves while another may still write to its inboxes
    if constexpr (DSM) cg::this_cluster().sync();
}

// Exclusive prefix of the per-row counts (one CTA); total -> *count.
__global__ void __launch_bounds__(1024) row_scan_kernel(const int* __restrict__ rowcnt, int H,
                                                        int* __restrict__ rowoff, int* count, const int* status) {
    if (*(volatile const int*)status & LOC_DEV_ERR_TIMEOUT) {   // the dithering gave up: no samples
        if (threadIdx.x == 0) *count = 0;
        return;
    }
    __shared__ int part[1024];
    const int per = (H + 1023) / 1024;
    const int j0 = threadIdx.x * per;
    int s = 0;
    for (int j = j0; j < j0 + per && j < H; ++j) s += rowcnt[j];
    part[threadIdx.x] = s;
    __syncthreads();
    for (int o = 1; o < 1024; o <<= 1) {            // inclusive Hillis-Steele scan
        const int v = threadIdx.x >= o ? part[threadIdx.x - o] : 0;
        __syncthreads();
        part[threadIdx.x] += v;
        __syncthreads();
    }
    int run = threadIdx.x > 0 ? part[threadIdx.x - 1] : 0;
    for (int j = j0; j < j0 + per && j < H; ++j) {
        rowoff[j] = run;
        run += rowcnt[j];
    }
    if (threadIdx.x == 1023) *count = part[1023];
}

// Selections as one byte a cell, for loc_dither's caller (with a loop over the bits on the host the call took
// 3.6 ms at 2048 x 2048, 2.0 like this).
__global__ void __launch_bounds__(NT) unpack_bits_kernel(const uint32_t* __restrict__ bits, size_t hw, int W,
                                                         uint8_t* __restrict__ out) {
    const int nch = (W + 31) / 32;
    for (size_t q = (size_t)blockIdx.x * NT + threadIdx.x; q < hw; q += (size_t)gridDim.x * NT) {
        const size_t j = q / W;
        const int i = (int)(q - j * W);
        out[q] = (bits[j * nch + (i >> 5)] >> (i & 31)) & 1u;
    }
}

// Linear indices of the selected cells in raster order (one warp per row, a word of 32 selections
// a lane), at most cap.
__global__ void __launch_bounds__(NT) compact_kernel(const uint32_t* __restrict__ selbits, const int* __restrict__ rowoff,
                                                     int H, int W, int cap, int32_t* __restrict__ out,
                                                     const int* status) {
    if (*(volatile const int*)status & LOC_DEV_ERR_TIMEOUT) return;   // no row offsets were made
    const int lane = threadIdx.x & 31, nch = (W + 31) / 32;
    for (int j = (blockIdx.x * NT + threadIdx.x) >> 5; j < H; j += (gridDim.x * NT) >> 5) {
        int base = rowoff[j];
        for (int c0 = 0; c0 < nch; c0 += 32) {
            uint32_t w = c0 + lane < nch ? selbits[(size_t)j * nch + c0 + lane] : 0u;
            const int n = __popc(w);
            int pos = n;                                       // inclusive prefix over the lanes
            for (int o = 1; o < 32; o <<= 1) {
                const int v = __shfl_up_sync(0xffffffffu, pos, o);
                if (lane >= o) pos += v;
            }
            const int total = __shfl_sync(0xffffffffu, pos, 31);
            pos += base - n;
            for (; w; w &= w - 1, ++pos)
                if (pos >= 0 && pos < cap) out[pos] = j * W + 32 * (c0 + lane) + __ffs(w) - 1;
            base += total;
        }
    }
}

// ------------------------------------------------------------------ ray casting + scoring

// Ranges for given cells and directions (the loc_ray_ranges entry point).
__global__ void __launch_bounds__(NT) ray_ranges_kernel(const uint8_t* __restrict__ trav, int H, int W,
                                                        const int32_t* __restrict__ cells, int n_cells,
                                                        const float* __restrict__ dirs, int n_dirs, float rmax,
                                                        float cell_m, float* __restrict__ out) {
    const size_t n = (size_t)n_cells * n_dirs;
    for (size_t q = (size_t)blockIdx.x * NT + threadIdx.x; q < n; q += (size_t)gridDim.x * NT) {
        const int c = (int)(q / n_dirs), d = (int)(q % n_dirs);
        const int cell = cells[c];
        const float t = dda_cells(trav, H, W, cell / W, cell % W, dirs[2 * d], dirs[2 * d + 1], rmax);
        out[q] = __fmul_rn(t, cell_m);
    }
}

// Order-preserving map of floats to unsigned ints (for atomicMax on floats).
__device__ __forceinline__ unsigned int f2ord(float f) {
    const unsigned int u = __float_as_uint(f);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float ord2f(unsigned int u) {
    return __uint_as_float((u & 0x80000000u) ? (u & 0x7FFFFFFFu) : ~u);
}

// The map as bits: bit b of word w of row j is 1 when cell (j, 32 w + b) is free (words per row
// wb = ceil(W / 32); bits past W are 0).
__global__ void __launch_bounds__(NT) pack_bits_kernel(const uint8_t* __restrict__ trav, int H, int W, int wb,
                                                       uint32_t* __restrict__ bits) {
    const size_t n = (size_t)H * wb;
    for (size_t q = (size_t)blockIdx.x * NT + threadIdx.x; q < n; q += (size_t)gridDim.x * NT) {
        const int j = (int)(q / wb), w = (int)(q % wb);
        uint32_t v = 0;
        for (int b = 0; b < 32; ++b) {
            const int i = 32 * w + b;
            if (i < W && trav[(size_t)j * W + i]) v |= 1u << b;
        }
        bits[q] = v;
    }
}

// One CTA per sampled cell (grid-stride): cast the n_dirs distinct rays once, then for every
// bin k: logL[s][k] = -sum_b (z_b - r(dir_of[k][b]))^2 / (2 sigma^2) over the used beams.
// With WIN the CTA first copies the map bits within R = ceil(rmax) + 2 cells of the sampled
// cell into shared memory (every cell a walk capped at rmax can look at), so each step of the
// walk reads shared memory instead of global memory; the walk itself is the same.
template <bool WIN>
__global__ void __launch_bounds__(kScoreNT) score_kernel(const uint8_t* __restrict__ trav, const uint32_t* __restrict__ bits,
                                                   int wb, int R, int wwin, int H, int W, int K,
                                                   const int32_t* __restrict__ samples, const int* count_ptr, int cap,
                                                   const float* __restrict__ dirs, int n_dirs,
                                                   const int32_t* __restrict__ dir_of, const float* __restrict__ z,
                                                   int n_used, float rmax, float cell_m, float inv2s2,
                                                   float* __restrict__ logL) {
    extern __shared__ float rh[];                 // n_dirs expected ranges (metres), then the window
    uint32_t* win = reinterpret_cast<uint32_t*>(rh + ((n_dirs + 3) & ~3));
    const int n = min(*count_ptr, cap);
    for (int s = blockIdx.x; s < n; s += gridDim.x) {
        const int cell = samples[s];
        const int j = cell / W, i = cell % W;
        if constexpr (WIN) {
            const int j0 = max(0, j - R), j1 = min(H - 1, j + R);
            const int w0 = max(0, i - R) >> 5, w1 = min(W - 1, i + R) >> 5;
            const int rows = j1 - j0 + 1, words = w1 - w0 + 1;
            for (int q = threadIdx.x; q < rows * words; q += kScoreNT) {
                const int r = q / words, c = q % words;
                win[r * wwin + c] = bits[(size_t)(j0 + r) * wb + w0 + c];
            }
            __syncthreads();
            const auto free_at = [win, j0, w0, wwin](int jj, int ii) {
                return ((win[(jj - j0) * wwin + ((ii >> 5) - w0)] >> (ii & 31)) & 1u) != 0u;
            };
            for (int d = threadIdx.x; d < n_dirs; d += kScoreNT)
                rh[d] = __fmul_rn(dda_walk(free_at, H, W, j, i, dirs[2 * d], dirs[2 * d + 1], rmax), cell_m);
        } else {
            for (int d = threadIdx.x; d < n_dirs; d += kScoreNT)
                rh[d] = __fmul_rn(dda_cells(trav, H, W, j, i, dirs[2 * d], dirs[2 * d + 1], rmax), cell_m);
        }
        __syncthreads();
        // one warp per bin: lane l sums the beams b = l, l + 32, ... in order, then a fixed
        // shuffle tree adds the lanes
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
        for (int k = warp; k < K; k += kScoreNT / 32) {
            const int32_t* row = dir_of + (size_t)k * n_used;
            float acc = 0.0f;
            for (int b = lane; b < n_used; b += 32) {
                const float e = z[b] - rh[row[b]];
                acc = fmaf(e, e, acc);
            }
            for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
            if (lane == 0) logL[(size_t)s * K + k] = -acc * inv2s2;
        }
        __syncthreads();
    }
}

// ------------------------------------------------------------------ Eq. 9 on the sampled set

struct ReweightScalars {
    double mass, wmass, factor;                   // sum b, sum b w over the set; mass / wmass
    unsigned int counter;
    int pad;
};

// Eq. 9 on the sampled set keeps its mass A = sum b and gives b' = A b L / sum(b L).  It is
// evaluated in the log domain against the offset c = max over the set of (log L + log b), so
// every weight w = exp(log L + log b - c) lies in (0, 1] with the largest equal to 1 and the
// normaliser sum w is at least 1: a scan whose likelihood peaks on states of tiny or zero
// belief cannot underflow the normaliser or overflow the factor.  States with b = 0 stay 0.
// reweight_max writes c (as an ordered uint; untouched when no state of the set holds mass).
template <typename T>
__global__ void __launch_bounds__(NT) reweight_max_kernel(const T* __restrict__ B, size_t hw, int K,
                                                          const int32_t* __restrict__ samples, const int* count_ptr,
                                                          int cap, const float* __restrict__ logL, unsigned int* maxL) {
    const int n = min(*count_ptr, cap);
    float best = -FLT_MAX;
    const size_t total = (size_t)n * K;
    for (size_t q = (size_t)blockIdx.x * NT + threadIdx.x; q < total; q += (size_t)gridDim.x * NT) {
        const int s = (int)(q / K), k = (int)(q % K);
        const float b = Store<T>::ld(B + (size_t)k * hw + samples[s]);
        if (b > 0.0f) best = fmaxf(best, logL[q] + logf(b));
    }
    for (int o = 16; o > 0; o >>= 1) best = fmaxf(best, __shfl_down_sync(0xffffffffu, best, o));
    if ((threadIdx.x & 31) == 0 && best > -FLT_MAX) atomicMax(maxL, f2ord(best));
}

// Sums over the sampled states (stored units): mass = sum b, wmass = sum w (the weights above);
// the last CTA writes factor = mass / wmass (0: leave the set as it is).
template <typename T>
__global__ void __launch_bounds__(NT) reweight_sums_kernel(const T* __restrict__ B, size_t hw, int K,
                                                           const int32_t* __restrict__ samples, const int* count_ptr,
                                                           int cap, const float* __restrict__ logL,
                                                           const unsigned int* maxL, double* partials,
                                                           ReweightScalars* rs) {
    __shared__ double red[NT / 32];
    __shared__ double red2[NT / 32];
    const int n = min(*count_ptr, cap);
    const double mx = (double)ord2f(*maxL);
    const bool any = isfinite(mx);                // some state of the set holds mass
    double m = 0.0, wm = 0.0;
    const size_t total = (size_t)n * K;
    for (size_t q = (size_t)blockIdx.x * NT + threadIdx.x; q < total && any; q += (size_t)gridDim.x * NT) {
        const int s = (int)(q / K), k = (int)(q % K);
        const double b = (double)Store<T>::ld(B + (size_t)k * hw + samples[s]);
        m += b;
        if (b > 0.0) wm += exp((double)logL[q] + log(b) - mx);
    }
    const double bm = block_sum<NT>(m, red);
    const double bw = block_sum<NT>(wm, red2);
    __shared__ int s_last;
    if (threadIdx.x == 0) {
        partials[2 * blockIdx.x] = bm;
        partials[2 * blockIdx.x + 1] = bw;
        __threadfence();
        s_last = atomicAdd(&rs->counter, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    double a = 0.0, c = 0.0;
    for (unsigned int b = threadIdx.x; b < gridDim.x; b += NT) {
        a += ((volatile double*)partials)[2 * b];
        c += ((volatile double*)partials)[2 * b + 1];
    }
    const double A = block_sum<NT>(a, red), C = block_sum<NT>(c, red2);
    if (threadIdx.x == 0) {
        rs->counter = 0u;
        rs->mass = A;
        rs->wmass = C;
        rs->factor = (C > 0.0 && isfinite(C) && A > 0.0) ? A / C : 0.0;
    }
}

// The new values b w factor of the sampled states, all (sample, bin) pairs in parallel: FP64
// exp and log, rounded to FP32 and written over logL (which they replace for the store below).
template <typename T>
__global__ void __launch_bounds__(NT) reweight_values_kernel(const T* __restrict__ B, size_t hw, int K,
                                                             const int32_t* __restrict__ samples,
                                                             const int* count_ptr, int cap, float* __restrict__ logL,
                                                             const unsigned int* maxL, const ReweightScalars* rs) {
    const double factor = rs->factor;
    if (!(factor > 0.0)) return;
    const int n = min(*count_ptr, cap);
    const double mx = (double)ord2f(*maxL);
    const size_t total = (size_t)n * K;
    for (size_t q = (size_t)blockIdx.x * NT + threadIdx.x; q < total; q += (size_t)gridDim.x * NT) {
        const int s = (int)(q / K), k = (int)(q % K);
        const size_t at = (size_t)k * hw + samples[s];
        // the new values sum to the set's old mass, so each is finite and at most that mass
        const double b = (double)Store<T>::ld(B + at);
        logL[q] = b > 0.0 ? (float)(factor * exp((double)logL[q] + log(b) - mx)) : 0.0f;
    }
}

// Stores the new values (one thread per sampled cell, its bins in order: the BF16 rounding
// residual runs along theta); the last CTA updates Z by the change of the set's sum.
template <typename T>
__global__ void __launch_bounds__(NT) reweight_apply_kernel(T* __restrict__ B, size_t hw, int K,
                                                            const int32_t* __restrict__ samples, const int* count_ptr,
                                                            int cap, const float* __restrict__ vals,
                                                            ReweightScalars* rs, double* partials, SessionDev* sd) {
    __shared__ double red[NT / 32];
    const double factor = rs->factor;
    const int n = min(*count_ptr, cap);
    KahanF acc;
    if (factor > 0.0) {
        for (int s = blockIdx.x * NT + threadIdx.x; s < n; s += gridDim.x * NT) {
            const size_t cell = (size_t)samples[s];
            const float* v = vals + (size_t)s * K;
            float res = 0.0f;
#pragma unroll 4
            for (int k = 0; k < K; ++k) acc.add(store_diffused<T>(B + (size_t)k * hw + cell, v[k], res));
        }
    }
    const double bt = block_sum<NT>(acc.value(), red);
    finish_sum<NT>(bt, partials, &sd->counter, gridDim.x, red, [sd, rs, factor](double S) {
        if (factor > 0.0) {
            const double Z = sd->Z - rs->mass + S;
            if (Z > 0.0 && isfinite(Z)) {
                sd->Z = Z;
                sd->inv_Z = (float)(1.0 / Z);
            }
        }
    });
}

unsigned int grid_for(size_t n, unsigned int cap) {
    size_t b = (n + NT - 1) / NT;
    if (b < 1) b = 1;
    return (unsigned int)(b < cap ? b : cap);
}

}  // namespace

size_t reweight_scalars_bytes() { return sizeof(ReweightScalars); }

#define LOC_DISPATCH(storage, CALL)                                                   \
    switch (storage) {                                                                \
        case LOC_F32: { using T = float; CALL; } break;                               \
        case LOC_BF16: { using T = __nv_bfloat16; CALL; } break;                      \
        case LOC_F16: { using T = __half; CALL; } break;                              \
        default: return cudaErrorInvalidValue;                                        \
    }

cudaError_t launch_belief_map(const void* B, int storage, const uint8_t* trav, SessionDev* sd, float inv_uniform,
                              int H, int W, int K, float* m, double* partials, unsigned int nparts,
                              unsigned int* counter, int n_samples, float* fs_out, cudaStream_t st) {
    const size_t hw = (size_t)H * W;
    const unsigned int nb = grid_for(hw, nparts < 2048 ? nparts : 2048);
    const size_t vec = storage == LOC_F32 ? 4 : 8;
    if (hw % vec == 0) {
        const unsigned int nbv = grid_for(hw / vec, nparts < 2048 ? nparts : 2048);
        LOC_DISPATCH(storage, (belief_map_vec_kernel<T, 16 / sizeof(T)><<<nbv, NT, 0, st>>>(
                                  (const T*)B, trav, sd, inv_uniform, hw, K, m, partials, counter, n_samples, fs_out)));
    } else {
        LOC_DISPATCH(storage, (belief_map_kernel<T><<<nb, NT, 0, st>>>((const T*)B, trav, sd, inv_uniform, hw, K, m,
                                                                          partials, counter, n_samples, fs_out)));
    }
    return cudaGetLastError();
}

cudaError_t launch_dither(const float* m, const float* fs, int H, int W, uint32_t* selbits, int* rowcnt, int* rowoff,
                          int* count, float* bnd, int* status, int cap, int32_t* samples, cudaStream_t st) {
    const int nrb = (H + 31) / 32;
    static PerDevice largest;                                  // cluster that the device can hold
    int dev = 0, max_ctas = 0;
    cudaGetDevice(&dev);
    cudaError_t e = largest.get(dev, &max_ctas, [](int* n) {
        const int most = (int)(kFsRingBytes + kFsInboxBytes);
        cudaError_t e = cudaSuccess;
        for (auto* f : {fs_kernel<true>, fs_kernel<false>}) {
            if (e == cudaSuccess) e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
            if (e == cudaSuccess) e = cudaFuncSetAttribute(f, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        }
        int fit = 0;
        for (*n = kFsMaxCtas; e == cudaSuccess && *n > 1; *n /= 2) {
            cudaLaunchConfig_t q{};
            cudaLaunchAttribute qa{};
            qa.id = cudaLaunchAttributeClusterDimension;
            qa.val.clusterDim.x = *n;
            qa.val.clusterDim.y = qa.val.clusterDim.z = 1;
            q.gridDim = dim3(*n);
            q.blockDim = dim3(kFsWarps * 64);
            q.dynamicSmemBytes = most;
            q.attrs = &qa;
            q.numAttrs = 1;
            if (cudaOccupancyMaxActiveClusters(&fit, fs_kernel<true>, &q) == cudaSuccess && fit > 0) break;
            cudaGetLastError();
        }
        return e;
    });
    if (e != cudaSuccess) return e;
    int ctas = 1;                                              // a power of two, one warp per block
    while (ctas < max_ctas && ctas * kFsWarps < nrb) ctas *= 2;
    // the inboxes in shared memory where the rows fit
    const int nbox = ctas * kFsWarps < nrb ? 2 : 1;
    const size_t boxes = sizeof(float) * kFsWarps * nbox * (size_t)((W + 31) / 32 * 32 + 64);
    const bool dsm = boxes <= kFsInboxBytes;
    const size_t smem = kFsRingBytes + (dsm ? boxes : 0);
    if (!dsm) e = cudaMemsetAsync(bnd, 0xFF, sizeof(float) * (size_t)nrb * W, st);   // kFsEmpty
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(ctas);
    cfg.blockDim = dim3(kFsWarps * 64);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = ctas;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    e = cudaLaunchKernelEx(&cfg, dsm ? fs_kernel<true> : fs_kernel<false>, m, fs, H, W, selbits, rowcnt, bnd, nbox, status);
    if (e != cudaSuccess) return e;
    row_scan_kernel<<<1, 1024, 0, st>>>(rowcnt, H, rowoff, count, status);
    if (samples)
        compact_kernel<<<grid_for((size_t)H * 32, 1024), NT, 0, st>>>(selbits, rowoff, H, W, cap, samples, status);
    return cudaGetLastError();
}

cudaError_t set_fs_wait(double seconds, int stall) {
    const unsigned long long ns = (unsigned long long)(seconds * 1e9);
    cudaError_t e = cudaMemcpyToSymbol(g_fs_wait_ns, &ns, sizeof(ns));
    if (e == cudaSuccess) e = cudaMemcpyToSymbol(g_fs_stall, &stall, sizeof(stall));
    return e;
}

cudaError_t launch_unpack_bits(const uint32_t* bits, int H, int W, uint8_t* out, cudaStream_t st) {
    unpack_bits_kernel<<<grid_for((size_t)H * W, 4096), NT, 0, st>>>(bits, (size_t)H * W, W, out);
    return cudaGetLastError();
}

cudaError_t launch_ray_ranges(const uint8_t* trav, int H, int W, const int32_t* cells, int n_cells, const float* dirs,
                              int n_dirs, float rmax_cells, float cell_m, float* out, cudaStream_t st) {
    ray_ranges_kernel<<<grid_for((size_t)n_cells * n_dirs, 4096), NT, 0, st>>>(trav, H, W, cells, n_cells, dirs,
                                                                              n_dirs, rmax_cells, cell_m, out);
    return cudaGetLastError();
}

cudaError_t launch_pack_bits(const uint8_t* trav, int H, int W, uint32_t* bits, cudaStream_t st) {
    const int wb = (W + 31) / 32;
    pack_bits_kernel<<<grid_for((size_t)H * wb, 4096), NT, 0, st>>>(trav, H, W, wb, bits);
    return cudaGetLastError();
}

cudaError_t launch_score_reweight(void* B, int storage, const uint8_t* trav, const uint32_t* bits, int H, int W, int K,
                                  const int32_t* samples, const int* count, int cap, const float* dirs, int n_dirs,
                                  const int32_t* dir_of, const float* z, int n_used, float rmax_cells, float cell_m,
                                  float inv2s2, float* logL, unsigned int* maxL, void* rs, double* partials,
                                  unsigned int nparts, SessionDev* sd, cudaStream_t st) {
    cudaError_t e = cudaMemsetAsync(maxL, 0, sizeof(unsigned int), st);
    if (e != cudaSuccess) return e;
    // the map window (R cells around the sampled cell) in shared memory when it fits
    const int R = (int)ceilf(rmax_cells) + 2;
    const int wwin = (2 * R + 1 + 31) / 32 + 1;
    const size_t rh_bytes = sizeof(float) * (size_t)((n_dirs + 3) & ~3);
    const size_t win_bytes = sizeof(uint32_t) * (size_t)(2 * R + 1) * wwin;
    const bool use_win = bits != nullptr && R < 4096 && rh_bytes + win_bytes <= kScoreWindowBytes;
    const size_t smem = rh_bytes + (use_win ? win_bytes : 0);
    // a grid-stride over the samples: CTAs past the count exit at once, but each still costs a launch
    const unsigned int ns = (unsigned int)(cap < 2048 ? (cap > 0 ? cap : 1) : 2048);
    const int wb = (W + 31) / 32;
    if (use_win) {
        if (smem > 48 * 1024) {
            e = cudaFuncSetAttribute(score_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
            if (e != cudaSuccess) return e;
        }
        score_kernel<true><<<ns, kScoreNT, smem, st>>>(trav, bits, wb, R, wwin, H, W, K, samples, count, cap, dirs, n_dirs,
                                                 dir_of, z, n_used, rmax_cells, cell_m, inv2s2, logL);
    } else {
        if (smem > 48 * 1024) {
            e = cudaFuncSetAttribute(score_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
            if (e != cudaSuccess) return e;
        }
        score_kernel<false><<<ns, kScoreNT, smem, st>>>(trav, bits, wb, R, wwin, H, W, K, samples, count, cap, dirs, n_dirs,
                                                  dir_of, z, n_used, rmax_cells, cell_m, inv2s2, logL);
    }
    const size_t hw = (size_t)H * W;
    const unsigned int half = nparts / 2 < 1024 ? nparts / 2 : 1024;
    const unsigned int nb = grid_for((size_t)cap * K, half > 0 ? half : 1);
    ReweightScalars* r = static_cast<ReweightScalars*>(rs);
    LOC_DISPATCH(storage, (reweight_max_kernel<T><<<nb, NT, 0, st>>>((const T*)B, hw, K, samples, count, cap, logL,
                                                                       maxL)));
    LOC_DISPATCH(storage, (reweight_sums_kernel<T><<<nb, NT, 0, st>>>((const T*)B, hw, K, samples, count, cap, logL,
                                                                        maxL, partials, r)));
    LOC_DISPATCH(storage, (reweight_values_kernel<T><<<nb, NT, 0, st>>>((const T*)B, hw, K, samples, count, cap, logL,
                                                                          maxL, r)));
    const unsigned int nb_cells = grid_for((size_t)cap, half > 0 ? half : 1);
    LOC_DISPATCH(storage, (reweight_apply_kernel<T><<<nb_cells, NT, 0, st>>>((T*)B, hw, K, samples, count, cap, logL,
                                                                               r, partials, sd)));
    return cudaGetLastError();
}

}  // namespace loc
