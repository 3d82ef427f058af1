// The streaming propagation (x/y radius 2, theta radius 3): Algorithm 1's propagation for all
// channels plus the Eq. 9 normaliser, one persistent CTA of 16 warps per SM.
//
// The CTA takes tiles of 28 x 64 output cells one after the other and streams their K planes.
// Its warps share nothing but mbarriers, so no barrier stops the whole CTA while planes flow:
//   * 1 manager warp fetches the next tile (its map mask into shared memory, two tiles deep)
//     and keeps one raw input box per blur warp in flight (TMA, the plane's shifted box);
//   * 8 blur warps, plane g of the stream going to warp g mod 8: bilinear shift, map mask and
//     x blur of the whole plane, S in registers only.  Lane r owns row r of the 32 halo rows
//     and walks along x, so the x blur needs no neighbour lane and S never meets memory;
//     rows are 4 mod 8 words apart, so the 16-byte loads of 8 lanes hit all 32 banks;
//   * 7 output warps (2 columns x 4 rows a thread): y blur into the register ring over theta,
//     theta blur, correction, store, normaliser and, with AM, the running argmax.
// The next tile's planes enter the pipeline while the output warps finish the previous tile.
//
// RAG: rows whose pitch is no multiple of 16 bytes.  TMA cannot address them, so each blur warp
// brings its own plane (load_rows); the stores are single values, and the operations follow the
// generic kernel's order, whose place it takes (613 x 797 x 48 FP32: 634 -> 79 us).
//
// Why this split.  The tile body it replaces ran S, X and P as passes of all warps through
// shared memory with two CTA barriers a plane: 42 to 53 thread instructions a cell and issue
// 41 to 52 % busy.  Here a cell costs 35 (FP32) to 39 (BF16), eight
// planes are in the works at once, and the latency of one plane's chain no longer counts.
// Every value is computed with the operations and the order of the passes in tiled_common.cuh, so
// tensors are those of the other tile configurations bit for bit.  A thread of the output warps sums
// its four rows before each compensated addition of the normaliser, as the synchronous configurations
// with four rows a thread do (two by two on ragged rows, as the generic kernel does).  Before and
// after, us a step: 64 x 64 x 16 FP32 27.3 -> 16.4, 500 x 500 x 128 111 -> 63, 512 x 512 x 64 63.5 -> 39.5,
// 1816 x 1816 x 36 FP16 310 -> 250, 2048 x 2048 x 72 BF16 725 -> 548 (2.2 TB/s) and FP32 793 -> 542 (4.5
// TB/s).  What bounds it now: the output warps' instruction issue and latency, two of them on a
// scheduler.
#pragma once
#include <type_traits>

#include "tiled_common.cuh"

namespace loc {
namespace stream {

using namespace tiled;

constexpr int TH = 28;                 // tile rows
constexpr int XR = TH + 2 * R;         // 32 rows of S and X: one per lane
constexpr int RAW_H = XR + 1;          // raw rows
constexpr int NB = 8;                  // blur warps = raw stages = X planes in flight
constexpr int NO = 7;                  // output warps
constexpr int NT = 32 * (1 + NB + NO); // 512
constexpr int SQ = 17;                 // quads of S columns (68 = 64 + 4)
constexpr int XPAD = 4;                // columns in front of an X row's 64
static_assert(XR == 32, "lane r of a blur warp owns row r");
// Warps 0 .. 6 are the output warps, 7 the manager, 8 .. 15 the blur warps: two warpgroups of
// each kind of register need.  The output warps' theta ring takes what the blur warps leave:
// 256 threads x (168 + 88) registers, at most the launch's 512 x kRegs (checked at set-up).
constexpr int kRegsOut = 168, kRegsBlur = 88, kRegs = (kRegsOut + kRegsBlur) / 2;

// raw box width: pitch 4 mod 8 words (conflict-free 16-byte loads down the rows)
template <typename T> constexpr int box_w() { return sizeof(T) == 4 ? 76 : 88; }

template <int V> using IC = std::integral_constant<int, V>;

struct OCfg {                          // rows of an output thread (2 columns each)
    static constexpr int MR = 4;
};

// One tile of work, as the manager hands it to the other warps.  K = 0: no more tiles.
struct Item {
    void* out;
    const void* in;                    // ragged rows only: X_{t-1}
    int reinit;                        // M is read in the place of X_{t-1}
    const uint8_t* trav;
    const float* corr;
    int K, H, W, ty0, tx0;
    float in_scale;
    float g0, g1, g2, gt[RING];
    int tile, ntiles;                  // index in its session, tiles of the session
    SessionDev* sd;
    double* partials;
    double log_out_mult;
};

template <typename T>
struct Smem {
    static constexpr int RAW = (RAW_H * box_w<T>() * (int)sizeof(T) + 127) / 128 * 128 / (int)sizeof(T);
    T raw[NB][RAW];                    // [RAW_H][box_w]
    float X[NB][XR][XW_PITCH];
    float wrap[NWRAP][TH][TW];
    float mk[2][XR][MW];
    Item item[2];
    int4 plan[2][LOC_MAX_K];           // each plane's source: first needed column, first row, fx, fy
    unsigned long long raw_full[NB], raw_empty[NB], x_full[NB], x_empty[NB], it_full[2], it_empty[2];
    double red[2][NO];                 // per item slot: the output warps' sums ...
    float am_v[2][NO];                 // ... and argmax candidates
    long long am_i[2][NO];
    volatile int fail;                 // a bounded wait gave up: every warp leaves its loop
    SessionDev* held;                  // QUEUE: session of the tile that the manager took but has not published
};

__device__ __forceinline__ void arrive(unsigned long long* b) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(su32(b)) : "memory");
}

// Wait of a whole warp, with the limit of bar_wait; false for every lane (and the CTA's fail
// flag set) when it ran out or another warp gave up.
template <typename SM>
__device__ __forceinline__ bool wait(SM& sm, unsigned long long* b, uint32_t parity) {
    bool ok = bar_try(b, parity);
    if (__all_sync(0xffffffffu, ok)) return true;
    ok = ok || (!sm.fail && bar_wait(b, parity));
    ok = __all_sync(0xffffffffu, ok);
    if (!ok) sm.fail = 1;
    return ok;
}

// Whether phase `parity` of b is complete, without waiting.
__device__ __forceinline__ bool bar_test(unsigned long long* b, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred q;\n mbarrier.test_wait.parity.shared::cta.b64 q, [%1], %2;\n"
        " selp.u32 %0, 1, 0, q;\n}\n"
        : "=r"(ok) : "r"(su32(b)), "r"(parity) : "memory");
    return ok != 0;
}

// S of four columns: raw columns e[0..4] of the lane's row (u) and of the next one (d), masked.
template <bool PACK>
__device__ __forceinline__ void s_quad(const float* u, const float* d, const float4 m, f2 fx2, f2 fy2, f2 gy2,
                                       float fx, float (&s)[4]) {
    f2 xu[2], xd[2];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const float u0 = u[2 * k], u1 = u[2 * k + 1], u2 = u[2 * k + 2];
        const float d0 = d[2 * k], d1 = d[2 * k + 1], d2 = d[2 * k + 2];
        if constexpr (PACK) {          // u0, u1 sit in an aligned register pair
            xu[k] = ffma2(fx2, pk(u1 - u0, u2 - u1), pk(u0, u1));
            xd[k] = ffma2(fx2, pk(d1 - d0, d2 - d1), pk(d0, d1));
        } else {
            xu[k] = pk(fmaf(fx, u1 - u0, u0), fmaf(fx, u2 - u1, u1));
            xd[k] = pk(fmaf(fx, d1 - d0, d0), fmaf(fx, d2 - d1, d1));
        }
    }
    const f2 o0 = fmul2(pk(m.x, m.y), ffma2(fy2, xd[0], fmul2(gy2, xu[0])));
    const f2 o1 = fmul2(pk(m.z, m.w), ffma2(fy2, xd[1], fmul2(gy2, xu[1])));
    upk(o0, s[0], s[1]);
    upk(o1, s[2], s[3]);
}

// X of four columns from S columns s[0..7].
__device__ __forceinline__ void x_quad(const float (&a)[4], const float (&b)[4], f2 g02, f2 g12, f2 g22, float* xp) {
    const f2 p0 = ffma2(g22, fadd2(pk(a[0], a[1]), pk(b[0], b[1])),
                        ffma2(g12, pk(a[1] + a[3], a[2] + b[0]), fmul2(g02, pk(a[2], a[3]))));
    const f2 p1 = ffma2(g22, fadd2(pk(a[2], a[3]), pk(b[2], b[3])),
                        ffma2(g12, pk(a[3] + b[1], b[0] + b[2]), fmul2(g02, pk(b[0], b[1]))));
    float v0, v1, v2, v3;
    upk(p0, v0, v1);
    upk(p1, v2, v3);
    *reinterpret_cast<float4*>(xp) = make_float4(v0, v1, v2, v3);
}

// The same in the order of the generic kernel (step_generic.cu), which grids of ragged rows took
// before: their tensors stay the same bit for bit.
__device__ __forceinline__ void s_quad_gen(const float* u, const float* d, const float4 m, float fx, float gx, f2 fy2,
                                           f2 gy2, float (&s)[4]) {
    float a[4], b[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        a[k] = __fmaf_rn(gx, u[k], __fmul_rn(fx, u[k + 1]));
        b[k] = __fmaf_rn(gx, d[k], __fmul_rn(fx, d[k + 1]));
    }
    const f2 o0 = fmul2(pk(m.x, m.y), ffma2(gy2, pk(a[0], a[1]), fmul2(fy2, pk(b[0], b[1]))));
    const f2 o1 = fmul2(pk(m.z, m.w), ffma2(gy2, pk(a[2], a[3]), fmul2(fy2, pk(b[2], b[3]))));
    upk(o0, s[0], s[1]);
    upk(o1, s[2], s[3]);
}
__device__ __forceinline__ void x_quad_gen(const float (&a)[4], const float (&b)[4], float g0, float g1, float g2,
                                           float* xp) {
    const float s[8] = {a[0], a[1], a[2], a[3], b[0], b[1], b[2], b[3]};
    float v[4];
#pragma unroll
    for (int k = 0; k < 4; ++k)
        v[k] = __fmaf_rn(g2, s[k + 4], __fmaf_rn(g1, s[k + 3], __fmaf_rn(g0, s[k + 2], __fmaf_rn(g1, s[k + 1], __fmul_rn(g2, s[k])))));
    *reinterpret_cast<float4*>(xp) = make_float4(v[0], v[1], v[2], v[3]);
}

// A 16-byte chunk of a raw row as floats.
template <typename T> struct Chunk;
template <> struct Chunk<float> {
    static constexpr int N = 4;
    static __device__ __forceinline__ void cvt(const uint4& r, float* v) {
        v[0] = __uint_as_float(r.x); v[1] = __uint_as_float(r.y);
        v[2] = __uint_as_float(r.z); v[3] = __uint_as_float(r.w);
    }
};
template <> struct Chunk<__nv_bfloat16> {
    static constexpr int N = 8;
    static __device__ __forceinline__ void cvt(const uint4& r, float* v) {
        const uint32_t w[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            v[2 * k] = __uint_as_float(w[k] << 16);
            v[2 * k + 1] = __uint_as_float(w[k] & 0xFFFF0000u);
        }
    }
};
template <> struct Chunk<__half> {
    static constexpr int N = 8;
    static __device__ __forceinline__ void cvt(const uint4& r, float* v) {
        const uint32_t w[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&w[k]));
            v[2 * k] = f.x;
            v[2 * k + 1] = f.y;
        }
    }
};

// Shift, mask and x blur of one plane: lane = row.  XO = the first needed column of the raw
// box (its residue in a 16-byte chunk).  The loads of chunk n + 2 are issued with chunk n; two
// chunks an iteration, so that the registers of the two chunks in hand change roles without
// moves and the eight alignments stay small enough for the instruction cache (fully unrolled,
// a third of the stalls were instruction fetches).
template <typename T, int XO, bool RAG>
__device__ __forceinline__ void blur_plane(const T* __restrict__ raw, const float* __restrict__ mk,
                                           float* __restrict__ X, float fx, float fy, f2 g02, f2 g12, f2 g22) {
    constexpr int N = Chunk<T>::N, BWT = box_w<T>(), QN = N / 4;      // QN S quads a chunk
    constexpr int CHUNKS = (SQ + QN - 1) / QN;                        // the last one needs its first quad only
    static_assert((CHUNKS & 1) == 1 && (CHUNKS + 2) * N <= BWT, "pairs of chunks and a last one; loads stay in the row");
    const int lane = threadIdx.x & 31;
    const uint4* up = reinterpret_cast<const uint4*>(raw + lane * BWT);
    const uint4* dn = reinterpret_cast<const uint4*>(raw + (lane + 1) * BWT);
    const float4* mp = reinterpret_cast<const float4*>(mk + lane * MW);
    float* xp = X + lane * XW_PITCH;
    const float gy = 1.0f - fy;
    const f2 fx2 = pk(fx, fx), fy2 = pk(fy, fy), gy2 = pk(gy, gy);
    constexpr bool PACK = (XO & 1) == 0;
    float ua[N], ub[N], da[N], db[N];               // chunks n and n + 1 of the row and of the next row
    uint4 un = up[1], dnx = dn[1];
    Chunk<T>::cvt(up[0], ua);
    Chunk<T>::cvt(dn[0], da);
    float s[4] = {0.f, 0.f, 0.f, 0.f}, t[4];
    float4 m = mp[0];
    // quad q of S from the raw columns of chunks (u, v) / (d, e), then X quad q - 1 from S quads
    // q - 1 and q (the first one, of no use, goes to the pad in front of the row)
    auto quad = [&](int q, int k, const float (&u)[N], const float (&v)[N], const float (&d)[N], const float (&e)[N],
                    float (&prev)[4], float (&now)[4]) {
        float w[5], z[5];
#pragma unroll
        for (int i = 0; i < 5; ++i) {
            const int c = XO + 4 * k + i;
            w[i] = c < N ? u[c] : v[c - N];
            z[i] = c < N ? d[c] : e[c - N];
        }
        const float4 mc = m;
        m = mp[q + 1];
        if constexpr (RAG) {
            float g0, g1, g2, dup;
            upk(g02, g0, dup);
            upk(g12, g1, dup);
            upk(g22, g2, dup);
            s_quad_gen(w, z, mc, fx, 1.0f - fx, fy2, gy2, now);
            x_quad_gen(prev, now, g0, g1, g2, xp + 4 * q);
        } else {
            s_quad<PACK>(w, z, mc, fx2, fy2, gy2, fx, now);
            x_quad(prev, now, g02, g12, g22, xp + 4 * q);
        }
    };
    // chunk n in (u, d); chunk n + 1 arrives in (v, e)
    auto chunk = [&](int n, const float (&u)[N], float (&v)[N], const float (&d)[N], float (&e)[N], float (&p)[4],
                     float (&q)[4]) {
        Chunk<T>::cvt(un, v);
        Chunk<T>::cvt(dnx, e);
        un = up[n + 2];
        dnx = dn[n + 2];
        quad(n * QN, 0, u, v, d, e, p, q);
        if constexpr (QN == 2) quad(n * QN + 1, 1, u, v, d, e, q, p);
    };
#pragma unroll 1
    for (int n = 0; n < CHUNKS - 1; n += 2) {
        chunk(n, ua, ub, da, db, s, t);
        if constexpr (QN == 2) chunk(n + 1, ub, ua, db, da, s, t);
        else chunk(n + 1, ub, ua, db, da, t, s);
    }
    Chunk<T>::cvt(un, ub);
    Chunk<T>::cvt(dnx, db);
    quad((CHUNKS - 1) * QN, 0, ua, ub, da, db, s, t);
}

template <typename T, bool RAG>
__device__ __forceinline__ void blur_any(const T* raw, const float* mk, float* X, int xo, float fx, float fy, f2 g0,
                                         f2 g1, f2 g2) {
    if constexpr (RAG) {               // the rows were placed by load_rows
        if (xo == 0) blur_plane<T, 0, true>(raw, mk, X, fx, fy, g0, g1, g2);
        else if constexpr (sizeof(T) == 2) blur_plane<T, 1, true>(raw, mk, X, fx, fy, g0, g1, g2);
        return;
    }
    switch (xo) {
        case 0: blur_plane<T, 0, false>(raw, mk, X, fx, fy, g0, g1, g2); break;
        case 1: blur_plane<T, 1, false>(raw, mk, X, fx, fy, g0, g1, g2); break;
        case 2: blur_plane<T, 2, false>(raw, mk, X, fx, fy, g0, g1, g2); break;
        case 3: blur_plane<T, 3, false>(raw, mk, X, fx, fy, g0, g1, g2); break;
        default:
            if constexpr (sizeof(T) == 2) {
                switch (xo) {
                    case 4: blur_plane<T, 4, false>(raw, mk, X, fx, fy, g0, g1, g2); break;
                    case 5: blur_plane<T, 5, false>(raw, mk, X, fx, fy, g0, g1, g2); break;
                    case 6: blur_plane<T, 6, false>(raw, mk, X, fx, fy, g0, g1, g2); break;
                    default: blur_plane<T, 7, false>(raw, mk, X, fx, fy, g0, g1, g2); break;
                }
            }
    }
}

// Ragged rows (a row pitch that is no multiple of 16 bytes, so no TMA): a blur warp brings its
// plane's box itself, rows y0 .. of plane p from column x, zeros outside the grid, without
// waiting (the caller waits for its asynchronous copies).  FP32, and 16-bit rows of even width,
// go as asynchronous 4-byte copies; 16-bit rows of odd width and a restart's map one element at
// a time, 24 loads in flight.  Returns the first needed column in the box.
template <typename T>
__device__ __forceinline__ int load_rows(T* raw, const Item& it, int p, int x, int y0) {
    const int lane = threadIdx.x & 31, H = it.H, W = it.W;
    constexpr int BWT = box_w<T>();
    const T* plane = static_cast<const T*>(it.in) + (size_t)p * H * W;
    if (it.reinit || (sizeof(T) == 2 && (W & 1))) {
        constexpr int COLS = 4 * SQ + 4;                       // 72: columns 0 .. 68 are needed
        for (int r0 = 0; r0 < RAW_H; r0 += 8) {
            T v[8][3];
#pragma unroll
            for (int r = 0; r < 8; ++r)
#pragma unroll
                for (int q = 0; q < 3; ++q) {
                    const int gy = y0 + r0 + r, gx = x + lane + 32 * q;
                    const bool in = r0 + r < RAW_H && gy >= 0 && gy < H && gx >= 0 && gx < W && lane + 32 * q < COLS;
                    const size_t at = in ? (size_t)gy * W + gx : 0;
                    v[r][q] = !in ? T(0.0f) : it.reinit ? T((float)it.trav[at]) : plane[at];
                }
#pragma unroll
            for (int r = 0; r < 8; ++r)
#pragma unroll
                for (int q = 0; q < 3; ++q)
                    if (r0 + r < RAW_H && lane + 32 * q < COLS) raw[(r0 + r) * BWT + lane + 32 * q] = v[r][q];
        }
        return 0;
    }
    constexpr int E = 4 / (int)sizeof(T);                      // elements a word
    constexpr int WORDS = (4 * SQ + 4) / E + (E > 1 ? 1 : 0), NW = (WORDS + 31) / 32;
    const int xo = x & (E - 1), xa = x - xo;
    const uint32_t dst = su32(raw) + 4 * lane;
    for (int r = 0; r < RAW_H; ++r) {
        const int gy = y0 + r;
        const bool row = gy >= 0 && gy < H;
        const T* src = plane + (row ? (size_t)gy * W : 0);
#pragma unroll
        for (int q = 0; q < NW; ++q) {
            const int wd = lane + 32 * q, gx = xa + E * wd;
            if (wd < WORDS) {
                const bool in = row && gx >= 0 && gx < W;
                asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(
                                 dst + (uint32_t)(r * BWT * sizeof(T) + 128 * q)),
                             "l"(in ? src + gx : plane), "r"(in ? 4 : 0)
                             : "memory");
            }
        }
    }
    return xo;
}

// A restart's input in place of a plane's TMA box, by its blur warp: the map (0 / 1) at columns x (a
// multiple of a 16-byte chunk) and rows y0 .. .  The grid's width is a multiple of 4 cells here, so a
// word of the map lies in the grid or outside it as a whole; four words a lane are in flight.  (With
// the manager warp filling every plane's box a cell at a time, a restart's step took 3.7 ms instead of
// 0.55 at 2048 x 2048 x 72 BF16; 0.69 like this.)
template <typename T>
__device__ __forceinline__ void load_map(T* raw, const Item& it, int x, int y0) {
    const int lane = threadIdx.x & 31, H = it.H, W = it.W;
    constexpr int BWT = box_w<T>(), WORDS = BWT / 4, ALL = RAW_H * WORDS;
    static_assert(BWT % 4 == 0, "whole words a row");
#pragma unroll 1
    for (int q0 = lane; q0 < ALL; q0 += 4 * 32) {
        uint32_t m[4];
#pragma unroll
        for (int n = 0; n < 4; ++n) {
            const int q = q0 + 32 * n, gy = y0 + q / WORDS, gx = x + 4 * (q % WORDS);
            m[n] = q < ALL && gy >= 0 && gy < H && gx >= 0 && gx < W
                       ? *reinterpret_cast<const uint32_t*>(it.trav + (size_t)gy * W + gx) : 0u;
        }
#pragma unroll
        for (int n = 0; n < 4; ++n) {
            const int q = q0 + 32 * n;
            struct alignas(4 * sizeof(T)) Four {
                T v[4];
            } o;
#pragma unroll
            for (int b = 0; b < 4; ++b) o.v[b] = T((float)((m[n] >> (8 * b)) & 0xFFu));
            if (q < ALL) *reinterpret_cast<Four*>(raw + 4 * q) = o;
        }
    }
}

// The manager's private side of a tile: where its planes come from.
struct Source {
    const CUtensorMap* tmap;
    const Shift* sh;
    int reinit;                        // the input is M (uniform restart): no TMA, the blur warps read it
};

// stall: the CTA's first (1) or second (2) tile is never handed over, since its barrier waits for one
// arrival more than comes (a test of the bounded waits); 0: none.
template <typename T>
__device__ __forceinline__ void init_barriers(Smem<T>& sm, int stall) {
    for (int s = 0; s < NB; ++s) {
        bar_init(&sm.raw_full[s], 1);
        bar_init(&sm.raw_empty[s], 1);
        bar_init(&sm.x_full[s], 1);
        bar_init(&sm.x_empty[s], NO);
    }
    for (int s = 0; s < 2; ++s) {
        bar_init(&sm.it_full[s], stall == s + 1 ? 2 : 1);
        bar_init(&sm.it_empty[s], NB + NO);
    }
    sm.fail = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

// The map mask over item t's halo region, by threads k of n.  The grid's width is a multiple of
// 4 cells (and device buffers are aligned to 16 bytes), so the map comes in whole words; W words a
// thread are in flight at once.
constexpr int MWORDS = 19;             // words a row: columns -4 .. 71 of the tile
template <int N, bool RAG, typename SM>
__device__ __forceinline__ void fill_mask(SM& sm, int slot, const Item& t, int k) {
    if constexpr (RAG) {               // byte loads
        constexpr int COLS = 4 * SQ;
#pragma unroll 8
        for (int q = k; q < XR * COLS; q += N) {
            const int r = q / COLS, c = q % COLS, y = t.ty0 - R + r, x = t.tx0 - R + c;
            sm.mk[slot][r][c] = y >= 0 && y < t.H && x >= 0 && x < t.W && t.trav[(size_t)y * t.W + x] ? 1.0f : 0.0f;
        }
        return;
    }
    constexpr int ALL = XR * MWORDS, W = (ALL + N - 1) / N;
    uint32_t m[W];
#pragma unroll
    for (int n = 0; n < W; ++n) {
        const int q = k + N * n, y = t.ty0 - R + q / MWORDS, x = t.tx0 - 4 + 4 * (q % MWORDS);
        m[n] = q < ALL && y >= 0 && y < t.H && x >= 0 && x < t.W
                   ? *reinterpret_cast<const uint32_t*>(t.trav + (size_t)y * t.W + x) : 0u;
    }
#pragma unroll
    for (int n = 0; n < W; ++n) {
        const int q = k + N * n, c = 4 * (q % MWORDS) - 2;    // halo column of the word
        if (q >= ALL) break;
        float* row = sm.mk[slot][q / MWORDS];
#pragma unroll
        for (int b = 0; b < 4; ++b)
            if (c + b >= 0) row[c + b] = (m[n] >> (8 * b)) & 0xFFu ? 1.0f : 0.0f;
    }
}

// The channel of plane p of the stream.  The outputs of planes 3 .. K-1, 0, 1, 2 are written in that
// order; for ragged rows the stream starts three channels earlier, so that they are written from
// channel 0 up, the order in which the generic kernel carries the BF16 residuals.
template <bool RAG>
__device__ __forceinline__ int channel(int p, int K) {
    return !RAG ? p : p >= RT ? p - RT : p - RT + K;
}

// Item t's plane sources into its slot, by lanes k of 32: many shift-table entries a load, so
// that issuing a plane waits for nothing but its stage (with a table read per plane the manager
// took ~1000 cycles a plane and was what bound the kernel).
template <bool RAG, typename SM>
__device__ __forceinline__ void fill_plan(SM& sm, int slot, const Item& t, const Source& from, int k) {
    for (int p = k; p < t.K; p += 32) {
        const Shift h = from.sh[channel<RAG>(p, t.K)];
        sm.plan[slot][p] = make_int4(t.tx0 - R + h.ox, t.ty0 - R + h.oy, __float_as_int(h.fx), __float_as_int(h.fy));
    }
}

// Manager warp, with the first item published in slot 0 (its plan too).  next(item, src) (all
// lanes, the same answer) gives the next tile or K = 0; done(item, slot) (all lanes) takes a
// finished tile's sums out of its slot.  QUEUE: the tiles are of several sessions, so the one in
// hand is kept for flag_failed.
template <typename T, bool RAG, bool QUEUE, typename Next, typename Done>
__device__ __forceinline__ void manage(Smem<T>& sm, Item it, Source src, Next next, Done done) {
    constexpr uint32_t kBoxBytes = RAW_H * box_w<T>() * sizeof(T);
    constexpr int AL = align_elems<T>();
    const int lane = threadIdx.x & 31;
    unsigned int g = 0;                // planes issued
    const int4* plan = sm.plan[0];
    // plane p of the tile in hand into the next raw stage
    auto issue = [&](int p) {
        const int s = g % NB;
        if (g >= NB && !wait(sm, &sm.raw_empty[s], ((g / NB) - 1) & 1)) return false;
        const int4 pl = plan[p];
        const int x_al = pl.x & ~(AL - 1), y0 = pl.y;
        if (lane == 0) {
            if (src.reinit) {          // the stage is the blur warp's, to fill with the map
                arrive(&sm.raw_full[s]);
            } else {
                bar_expect(&sm.raw_full[s], kBoxBytes);
                tma_load(&sm.raw[s][0], src.tmap, &sm.raw_full[s], x_al, y0, p);
            }
        }
        ++g;
        return true;
    };
    // item i is finished: its sums leave the slot
    auto retire = [&](unsigned int i) {
        const int slot = i & 1;
        if (!wait(sm, &sm.it_empty[slot], (i >> 1) & 1)) return false;
        done(sm.item[slot], slot);
        __syncwarp();
        return true;
    };
    auto publish = [&](unsigned int i, const Item& t, const Source& from) {
        const int slot = i & 1;
        if (i >= 2 && !retire(i - 2)) return false;
        if (t.K) {
            fill_plan<RAG>(sm, slot, t, from, lane);
            fill_mask<32, RAG>(sm, slot, t, lane);
        }
        if (lane == 0) {
            sm.item[slot] = t;
            if constexpr (QUEUE) sm.held = nullptr;
        }
        __syncwarp();
        if (lane == 0) arrive(&sm.it_full[slot]);
        return true;
    };
    auto take = [&](Item& t, Source& from) {
        next(t, from);
        if constexpr (QUEUE) {
            if (lane == 0 && t.K) sm.held = t.sd;
        }
    };
    bool ok = true;
    unsigned int i = 0;
    for (; ok && it.K; ++i) {
        Item nit{};
        Source nsrc{};
        if constexpr (RAG) {           // the blur warps bring the planes
            take(nit, nsrc);
            ok = publish(i + 1, nit, nsrc);
        } else for (int p = 0; ok && p < it.K; ++p) {
            ok = issue(p);
            if (ok && p == (it.K > NB ? NB : it.K - 1)) {   // early in the tile: the next one
                take(nit, nsrc);
                ok = publish(i + 1, nit, nsrc);
            }
        }
        it = nit;
        src = nsrc;
        plan = sm.plan[(i + 1) & 1];
    }
    if (ok && i) ok = retire(i - 1);   // the last tile (the one before went with its successor)
    if (!ok) {
        // let the copies in flight land (bounded) before the CTA may leave
        for (unsigned int q = g > NB ? g - NB : 0; q < g; ++q) bar_wait(&sm.raw_full[q % NB], (q / NB) & 1);
    }
}

template <typename T, bool RAG>
__device__ __forceinline__ void blur(Smem<T>& sm, int w) {
    const int lane = threadIdx.x & 31;
    unsigned int g = w, base = 0;
    for (unsigned int i = 0;; ++i) {
        const int slot = i & 1;
        if (!wait(sm, &sm.it_full[slot], (i >> 1) & 1)) return;
        const Item& it = sm.item[slot];
        const unsigned int K = it.K;
        if (K == 0) return;
        const bool restart = !RAG && it.reinit;
        const f2 g0 = pk(it.g0, it.g0), g1 = pk(it.g1, it.g1), g2 = pk(it.g2, it.g2);
        for (; g < base + K; g += NB) {
            const uint32_t ph = (g / NB) & 1;
            const int4 pl = sm.plan[slot][g - base];
            int xo;
            if constexpr (RAG) xo = load_rows<T>(sm.raw[w], it, channel<true>(g - base, K), pl.x, pl.y);
            else xo = pl.x & (align_elems<T>() - 1);
            if constexpr (!RAG) {
                if (restart) {
                    if (!wait(sm, &sm.raw_full[w], ph)) return;
                    load_map<T>(sm.raw[w], it, pl.x - xo, pl.y);
                    __syncwarp();
                }
            }
            if (g >= NB && !wait(sm, &sm.x_empty[w], ph ^ 1)) return;
            if constexpr (RAG) {
                asm volatile("cp.async.wait_all;" ::: "memory");
                __syncwarp();
            } else if (!wait(sm, &sm.raw_full[w], ph)) {
                return;
            }
            blur_any<T, RAG>(sm.raw[w], &sm.mk[slot][0][0], &sm.X[w][0][0], xo, __int_as_float(pl.z),
                             __int_as_float(pl.w), g0, g1, g2);
            // the stage that plain stores wrote may take a TMA copy next
            if (restart) asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncwarp();
            if (lane == 0) {
                if constexpr (!RAG) arrive(&sm.raw_empty[w]);
                arrive(&sm.x_full[w]);
            }
        }
        __syncwarp();
        if (lane == 0) arrive(&sm.it_empty[slot]);
        base += K;
    }
}

// The stored form of two neighbouring outputs and its value as FP32: FP32 as is, BF16 by error
// diffusion along theta, FP16 to nearest (see store2).
template <typename T> __device__ __forceinline__ f2 put2(T* p, f2 v, f2& res, bool on);
// Two outputs of a ragged row: no alignment, each column with its own guard (on0, on1).
template <typename T>
__device__ __forceinline__ f2 put1(T* p, f2 v, f2& res, bool on0, bool on1) {
    T tmp[2];
    f2 st;
    float a, b;
    upk(v, a, b);
    if constexpr (std::is_same_v<T, __nv_bfloat16>) {
        const uint32_t d = bf16x2_diffuse(a, b, res, st);
        tmp[0] = __ushort_as_bfloat16((unsigned short)d);
        tmp[1] = __ushort_as_bfloat16((unsigned short)(d >> 16));
    } else if constexpr (std::is_same_v<T, __half>) {
        tmp[0] = __float2half_rn(a);
        tmp[1] = __float2half_rn(b);
        st = pk(__half2float(tmp[0]), __half2float(tmp[1]));
    } else {
        tmp[0] = a;
        tmp[1] = b;
        st = v;
    }
    if (on0) p[0] = tmp[0];
    if (on1) p[1] = tmp[1];
    return st;
}
template <> __device__ __forceinline__ f2 put2<float>(float* p, f2 v, f2&, bool on) {
    if (on) *reinterpret_cast<f2*>(p) = v;
    return v;
}
template <> __device__ __forceinline__ f2 put2<__nv_bfloat16>(__nv_bfloat16* p, f2 v, f2& res, bool on) {
    float a, b;
    f2 st;
    upk(v, a, b);
    const uint32_t d = bf16x2_diffuse(a, b, res, st);
    if (on) *reinterpret_cast<uint32_t*>(p) = d;
    return st;
}
template <> __device__ __forceinline__ f2 put2<__half>(__half* p, f2 v, f2&, bool on) {
    float a, b;
    upk(v, a, b);
    const __half2 h = __floats2half2_rn(a, b);
    if (on) *reinterpret_cast<__half2*>(p) = h;
    return pk(__low2float(h), __high2float(h));
}

// A thread's best positive stored value so far and the plane it lies in (lowest plane on ties).
struct PlaneBest {
    float v = 0.0f;
    int o = INT_MAX;
};

// A thread's best plane as a value and linear index: its stored values of that plane are read
// back (the thread's own writes) and the first one equal to the value is taken.
template <typename T>
__device__ __forceinline__ ArgBest locate(const Item& it, int t, const PlaneBest& b) {
    ArgBest r;
    float top = b.v;                                     // only the warp's best threads look
    for (int o = 16; o > 0; o >>= 1) top = fmaxf(top, __shfl_xor_sync(0xffffffffu, top, o));
    if (b.v != top || b.o == INT_MAX) return r;
    const T* plane = static_cast<const T*>(it.out) + (size_t)b.o * it.H * it.W;
    for (int rr = OCfg::MR - 1; rr >= 0; --rr)
        for (int c = 1; c >= 0; --c) {
            const int gy = it.ty0 + OCfg::MR * (t >> 5) + rr, gx = it.tx0 + 2 * (t & 31) + c;
            if (gy < it.H && gx < it.W && Store<T>::ld(plane + (size_t)gy * it.W + gx) == b.v) {
                r.v = b.v;
                r.i = ((long long)b.o * it.H + gy) * it.W + gx;
            }
        }
    return r;
}

// Output warps: a tile's sums (and argmax candidates) go to its slot, for the manager.
//
// Per plane: the X rows of plane p + 1 are loaded before the theta blur and the stores of
// plane p, and its y blur follows them, so eight independent chains hide the latencies; runs
// of 7 planes away from the ends carry no conditions.  Outside the grid the correction is 0,
// so only the stores are guarded.
template <typename T, bool AM, bool RAG>
__device__ __forceinline__ void output(Smem<T>& sm, int t) {
    constexpr int MR = OCfg::MR;
    const int lane = t & 31, r0 = MR * (t >> 5);
    unsigned int base = 0;
    for (unsigned int i = 0;; ++i) {
        const int slot = i & 1;
        if (!wait(sm, &sm.it_full[slot], (i >> 1) & 1)) return;
        const Item& it = sm.item[slot];
        const int K = it.K;
        if (K == 0) return;
        const int gx = it.tx0 + 2 * lane;
        f2 cs[MR];
        bool on[MR];
        T* out[MR];                                      // the thread's rows in the plane to write
        const size_t plane = (size_t)it.H * it.W;
#pragma unroll
        for (int rr = 0; rr < MR; ++rr) {
            const int gy = it.ty0 + r0 + rr;
            on[rr] = gy < it.H && gx < it.W;
            const size_t at = (size_t)gy * it.W + gx;
            out[rr] = static_cast<T*>(it.out) + (RAG ? 0 : RT * plane) + at;   // the first channel written
            float c0 = 0.0f, c1 = 0.0f;
            if (on[rr]) {
                c0 = it.corr[at] * it.in_scale;
                if (!RAG || gx + 1 < it.W) c1 = it.corr[at + 1] * it.in_scale;
            }
            cs[rr] = pk(c0, c1);
        }
        const bool pair = !RAG || gx + 1 < it.W;         // the second column is in the grid too
        const f2 g0 = pk(it.g0, it.g0), g1 = pk(it.g1, it.g1), g2 = pk(it.g2, it.g2);
        f2 gt[RT + 1];                                   // symmetric taps: centre, +-1, +-2, +-3
#pragma unroll
        for (int d = 0; d <= RT; ++d) gt[d] = pk(it.gt[RT + d], it.gt[RT + d]);
        f2 ring[RING][MR], res[MR], x[MR + 4];
#pragma unroll
        for (int k = 0; k < MR; ++k) res[k] = 0ull;
        KahanF2 acc;
        PlaneBest best;
        bool ok = true;
        // X rows of plane p.  The barrier of the plane after it is tested here, so that its answer
        // is there when that plane's turn comes (a wait at that point cost ~100 cycles a plane
        // with the data long ready).
        bool ready = false;
        auto load = [&](int p) {
            const unsigned int g = base + (unsigned int)p, h = g + 1;
            if (!__all_sync(0xffffffffu, ready)) ok &= wait(sm, &sm.x_full[g % NB], (g / NB) & 1);
            const float* xr = &sm.X[g % NB][r0][XPAD + 2 * lane];
#pragma unroll
            for (int q = 0; q < MR + 4; ++q) x[q] = *reinterpret_cast<const f2*>(xr + q * XW_PITCH);
            ready = bar_test(&sm.x_full[h % NB], (h / NB) & 1);
        };
        // their y blur into ring slot PH
        auto yblur = [&](int p, auto ph) {
            constexpr int PH = decltype(ph)::value;
#pragma unroll
            for (int rr = 0; rr < MR; ++rr)
                ring[PH][rr] = RAG ? ffma2(g2, x[rr + 4], ffma2(g1, x[rr + 3], ffma2(g0, x[rr + 2], ffma2(g1, x[rr + 1], fmul2(g2, x[rr])))))
                                   : ffma2(g2, fadd2(x[rr], x[rr + 4]), ffma2(g1, fadd2(x[rr + 1], x[rr + 3]), fmul2(g0, x[rr + 2])));
            __syncwarp();
            if (lane == 0) arrive(&sm.x_empty[(base + (unsigned int)p) % NB]);
        };
        // output plane o, the ring holding planes o - 3 .. o + 3 with the newest in slot PH
        auto theta = [&](int o, auto ph) {
            constexpr int PH = decltype(ph)::value;
            f2 st[MR];
#pragma unroll
            for (int rr = 0; rr < MR; ++rr) {
                f2 v = fmul2(gt[RT], ring[(PH + 1) % RING][rr]);
#pragma unroll
                for (int d = 1; d < RING; ++d) v = ffma2(gt[d < RT ? RT - d : d - RT], ring[(PH + 1 + d) % RING][rr], v);
                if constexpr (RAG) st[rr] = put1<T>(out[rr], fmul2(cs[rr], v), res[rr], on[rr], on[rr] && pair);
                else st[rr] = put2<T>(out[rr], fmul2(cs[rr], v), res[rr], on[rr]);
                out[rr] += plane;
            }
            if constexpr (RAG) {                         // two values a compensated addition, as the generic kernel
                static_assert(MR % 2 == 0, "pairs of rows");
#pragma unroll
                for (int rr = 0; rr < MR; rr += 2) acc.add(fadd2(st[rr], st[rr + 1]));
            } else {
                f2 part = st[0];
#pragma unroll
                for (int rr = 1; rr < MR; ++rr) part = fadd2(part, st[rr]);
                acc.add(part);
            }
            if constexpr (AM) {
                float m = -FLT_MAX;
#pragma unroll
                for (int rr = 0; rr < MR; ++rr) {
                    float lo, hi;
                    upk(st[rr], lo, hi);
                    m = fmaxf(m, fmaxf(lo, hi));
                }
                if (m > best.v || (m == best.v && o < best.o)) {
                    best.v = m;
                    best.o = o;
                }
            }
        };
        // planes 0 .. 5: also kept for the circular end
        auto head = [&](int p, auto ph) {
            constexpr int PH = decltype(ph)::value;
            load(p);
            yblur(p, ph);
#pragma unroll
            for (int rr = 0; rr < MR; ++rr) *reinterpret_cast<f2*>(&sm.wrap[PH][r0 + rr][2 * lane]) = ring[PH][rr];
        };
        head(0, IC<0>{});
        head(1, IC<1>{});
        head(2, IC<2>{});
        head(3, IC<3>{});
        head(4, IC<4>{});
        head(5, IC<5>{});
        load(6);
        yblur(6, IC<6>{});
        // step p writes plane p - 3 and brings plane p + 1 into the ring
        auto step = [&](int p, auto ph) {
            constexpr int PH = decltype(ph)::value;
            load(p + 1);
            theta(p - RT, ph);
            yblur(p + 1, IC<(PH + 1) % RING>{});
        };
        auto tail = [&](int p, auto ph) {
            constexpr int PH = decltype(ph)::value, NX = (PH + 1) % RING;
            if (p >= K + NWRAP) return;
            if (!RAG && p - RT == K) {                   // the last planes written are 0, 1, 2
#pragma unroll
                for (int rr = 0; rr < MR; ++rr) out[rr] -= (size_t)K * plane;
            }
            const int o = p - RT < K ? p - RT : p - RT - K;
            if (p + 1 < K) load(p + 1);
            theta(o, ph);
            if (p + 1 < K) {
                yblur(p + 1, IC<NX>{});
            } else if (p + 1 < K + NWRAP) {
#pragma unroll
                for (int rr = 0; rr < MR; ++rr)
                    ring[NX][rr] = *reinterpret_cast<const f2*>(&sm.wrap[p + 1 - K][r0 + rr][2 * lane]);
            }
        };
        int p = RING - 1;
        for (; p + RING < K; p += RING) {
            step(p, IC<6>{});
            step(p + 1, IC<0>{});
            step(p + 2, IC<1>{});
            step(p + 3, IC<2>{});
            step(p + 4, IC<3>{});
            step(p + 5, IC<4>{});
            step(p + 6, IC<5>{});
        }
        for (; p < K + NWRAP; p += RING) {
            tail(p, IC<6>{});
            tail(p + 1, IC<0>{});
            tail(p + 2, IC<1>{});
            tail(p + 3, IC<2>{});
            tail(p + 4, IC<3>{});
            tail(p + 5, IC<4>{});
            tail(p + 6, IC<5>{});
        }
        if (!__all_sync(0xffffffffu, ok)) return;
        double v = acc.value();
        for (int q = 16; q > 0; q >>= 1) v += __shfl_down_sync(0xffffffffu, v, q);
        if (lane == 0) sm.red[slot][t >> 5] = v;
        if constexpr (AM) {
            ArgBest b = locate<T>(it, t, best);
            for (int q = 16; q > 0; q >>= 1) {
                const float ov = __shfl_down_sync(0xffffffffu, b.v, q);
                const long long oi = __shfl_down_sync(0xffffffffu, b.i, q);
                if (am_better(ov, oi, b.v, b.i)) {
                    b.v = ov;
                    b.i = oi;
                }
            }
            if (lane == 0) {
                sm.am_v[slot][t >> 5] = b.v;
                sm.am_i[slot][t >> 5] = b.i;
            }
        }
        __syncwarp();
        if (lane == 0) arrive(&sm.it_empty[slot]);
        base += (unsigned int)K;
    }
}

// The manager's end of a tile: its partial and, with AM, its argmax candidate go to p / pv / pi
// [it.tile]; the tile that arrives last at `counter` combines all `ntiles` of them in a fixed
// order and calls fin(sum, best) from lane 0.
template <bool AM, typename SM, typename Fin>
__device__ __forceinline__ void retire_tile(const SM& sm, const Item& it, int slot, double* p, float* pv,
                                            long long* pi, unsigned int* counter, Fin fin) {
    const int lane = threadIdx.x & 31;
    int last = 0;
    if (lane == 0) {
        double v = 0.0;
        for (int w = 0; w < NO; ++w) v += sm.red[slot][w];
        p[it.tile] = v;
        if constexpr (AM) {
            ArgBest b;
            for (int w = 0; w < NO; ++w)
                if (am_better(sm.am_v[slot][w], sm.am_i[slot][w], b.v, b.i)) {
                    b.v = sm.am_v[slot][w];
                    b.i = sm.am_i[slot][w];
                }
            pv[it.tile] = b.v;
            pi[it.tile] = b.i;
        }
        __threadfence();
        last = atomicAdd(counter, 1u) == (unsigned int)(it.ntiles - 1);
    }
    if (!__shfl_sync(0xffffffffu, last, 0)) return;
    __threadfence();
    double s = 0.0;
    ArgBest b;
#pragma unroll 4
    for (int q = lane; q < it.ntiles; q += 32) {
        s += ((volatile double*)p)[q];
        if constexpr (AM) {
            const float v = ((volatile float*)pv)[q];
            const long long i = ((volatile long long*)pi)[q];
            if (am_better(v, i, b.v, b.i)) {
                b.v = v;
                b.i = i;
            }
        }
    }
    for (int q = 16; q > 0; q >>= 1) {
        s += __shfl_down_sync(0xffffffffu, s, q);
        if constexpr (AM) {
            const float v = __shfl_down_sync(0xffffffffu, b.v, q);
            const long long i = __shfl_down_sync(0xffffffffu, b.i, q);
            if (am_better(v, i, b.v, b.i)) {
                b.v = v;
                b.i = i;
            }
        }
    }
    if (lane == 0) {
        *counter = 0u;
        fin(s, b);
    }
}

// QUEUE, before run_roles, by one thread: no tile in the second slot (the first gets one before any wait)
// and none in the manager's hands.
template <typename SM>
__device__ __forceinline__ void none_taken(SM& sm) {
    sm.item[1].K = 0;
    sm.held = nullptr;
}
// QUEUE, after run_roles, by one thread of a CTA that gave up: flags the sessions of every tile that it
// took and whose sums it did not record, which are those in the slots and the one in the manager's hands.
template <typename SM>
__device__ __forceinline__ void flag_failed(const SM& sm) {
    for (int k = 0; k < 2; ++k)
        if (sm.item[k].K > 0) atomicOr(&sm.item[k].sd->status, LOC_DEV_ERR_TIMEOUT);
    if (sm.held) atomicOr(&sm.held->status, LOC_DEV_ERR_TIMEOUT);
}

// The roles of the CTA's warps; next and done as for manage(), stall as for init_barriers().  next()
// gives a tile's geometry and input(item, src) what earlier work on the stream wrote (scale, restart
// flag); for the first tile begin() runs between them, the barriers, the plan and the map mask being
// set up by then: the manager's planes travel while the other warps read the map.
template <typename T, bool AM, bool RAG, bool QUEUE, typename Next, typename Begin, typename Input, typename Done>
__device__ __forceinline__ void run_roles(Smem<T>& sm, int stall, Next next, Begin begin, Input input, Done done) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    Item it{};
    Source src{};
    if (warp == NO) {
        next(it, src);
        if (lane == 0) {
            init_barriers(sm, stall);
            sm.item[0] = it;
        }
        fill_plan<RAG>(sm, 0, it, src, lane);
    }
    __syncthreads();
    if (warp != NO) {
        const Item& t = sm.item[0];
        if (t.K) fill_mask<NT - 32, RAG>(sm, 0, t, warp < NO ? threadIdx.x : threadIdx.x - 32);
        asm volatile("bar.sync 1, %0;" ::"n"(NT - 32) : "memory");
    } else {
        begin();
        input(it, src);
        if (lane == 0) {
            sm.item[0].in_scale = it.in_scale;
            sm.item[0].reinit = it.reinit;
            arrive(&sm.it_full[0]);
        }
        __syncwarp();
    }
    if (warp < NO + 1) {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kRegsOut));
        if (warp < NO) output<T, AM, RAG>(sm, threadIdx.x);
        else manage<T, RAG, QUEUE>(sm, it, src, [&](Item& t, Source& s) {
            next(t, s);
            input(t, s);
        }, done);
    } else {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kRegsBlur));
        blur<T, RAG>(sm, warp - (NO + 1));
    }
    __syncthreads();
}

// Dynamic shared memory and the register split of kernel f: the limit is set, and the launch's
// registers must cover the split (a warpgroup would wait for registers that never come).
template <typename T, typename F>
cudaError_t prepare(F f) {
    cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(Smem<T>) + 128);
    cudaFuncAttributes at{};
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&at, f);
    if (e == cudaSuccess && at.numRegs < kRegs) e = cudaErrorInvalidConfiguration;
    return e;
}

// The session scalars from the new normaliser Z (Eq. 9): Z, 1/Z and the log-scale, or the
// uniform restart when no mass is left.
__device__ __forceinline__ void session_finish(SessionDev* sd, double Z, double log_mult) {
    sd->n_prop += 1;
    if (Z > 0.0 && isfinite(Z)) {
        sd->Z = Z;
        sd->inv_Z = (float)(1.0 / Z);
        sd->logscale += log(Z) - log_mult;
        sd->reinit = 0;
    } else {
        if (!isfinite(Z)) sd->status |= LOC_DEV_ERR_NONFINITE_Z;
        sd->Z = 1.0;
        sd->inv_Z = 1.0f;
        sd->reinit = 1;
        sd->n_reinit += 1;
    }
}

}  // namespace stream
}  // namespace loc
