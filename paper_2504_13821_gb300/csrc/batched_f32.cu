// The FP32 kernel of the batched uneven problems (batched.cu has the FP64 one and
// the launch): one persistent launch whose CTAs take the problems, largest first,
// from an atomic counter. A problem runs in chunks of 16, 32 or 64 right-hand sides
// held in shared memory (k rows x W columns); M passes through shared memory once
// per chunk, 16 columns at a time.
//
//   TRSM, right-looking in 16-row blocks: substitution on the block (a lane per
//     column, on a tile that arrived during the block before), while the block's
//     columns of M below it arrive by cp.async; then every row below takes the
//     rank-16 update in register tiles of 8, 4 or 2 rows x 4 columns;
//   TRMM, row bands from the bottom: a band's rows accumulate over their K range
//     16 columns of M at a time in the same tiles, then replace their own rows of
//     the chunk (no row above reads them).
//
// What bounds it: the chain of a chunk's blocks (one of order 512 and 32 columns alone
// on the GPU takes 2.2 us per block: 0.9 for the columns of M to arrive, 0.6 for the
// substitution, 1.2 for the update, in part at once), which two CTAs per SM hide in
// part; the FMA pipe is 27 % active. 4096 problems of order 16..512 with 1..64 right-hand
// sides: 955 us with the kernel before it (M read four scalar loads to 16 FMAs through
// L1, 32 columns only, a CTA a problem, FMA pipe 20 % active), 491 with this one
// (1000 problems: 673 -> 164, 200: 361 -> 84).
#include "batched.cuh"
#include "common.cuh"

namespace trx {
namespace {

constexpr int NT = 256, SB = 16, MAXK = kBatchOrder;
template <int W>
constexpr int LDC = W + 4;                             // row stride of the chunk
constexpr int LDB = 256 + 4;                           // row stride of a TRMM band's columns
// Floats for the chunk and M's columns: two CTAs per SM with the rest.
constexpr int SPACE = (115200 / 4 - 2 * SB * SB - MAXK) / 4 * 4;
constexpr size_t SMEM = sizeof(float) * (SPACE + 2 * SB * SB + MAXK);
static_assert(MAXK * LDC<32> + SB * (MAXK - SB + 8 + 4) <= SPACE, "one panel beside the chunk");
static_assert(256 * LDC<64> + SB * (256 - SB + 8 + 4) <= SPACE, "64-column chunks up to order 256");
static_assert(MAXK * LDC<32> + 2 * SB * LDB <= SPACE && 256 * LDC<64> + 2 * SB * LDB <= SPACE,
              "two buffers of a TRMM band beside the chunk");

__device__ __forceinline__ uint64_t pack2(float a, float b) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ void unpack2(uint64_t r, float& a, float& b) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(r));
}
__device__ __forceinline__ uint64_t ffma2(uint64_t a, uint64_t b, uint64_t c) {
    uint64_t d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}

// One problem's view: M(i, l) = A[i * rs + l * cs].
struct View {
    const float* A;
    int64_t rs, cs;
    int k;
    bool row_fast;
};

// One float global -> shared, asynchronous.
__device__ __forceinline__ void cp_async4(uint32_t dst, const float* src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async4_if(uint32_t dst, const float* src, bool on) {
    asm volatile(
        "{ .reg .pred p; setp.ne.b32 p, %2, 0; @p cp.async.ca.shared.global [%0], [%1], 4; }" ::"r"(
            dst),
        "l"(src), "r"((int)on)
        : "memory");
}
__device__ __forceinline__ void cp_async_commit() {
    asm volatile("cp.async.commit_group;" ::: "memory");
}
template <int N>
__device__ __forceinline__ void cp_async_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// Elements 0, 32, 64, ... below n of a contiguous run in direction DIR, STEP words
// apart in shared memory: constant steps, so a copy costs little more than its own
// instruction (with a 64-bit product per element, staging was a third of all
// instructions).
template <int DIR, int STEP>
__device__ __forceinline__ void stage_run(const float* src, uint32_t dst, int n) {
    for (; n > 0; n -= 128, src += 128 * DIR, dst += 16 * STEP)
#pragma unroll
        for (int u = 0; u < 4; ++u) cp_async4_if(dst + 4 * STEP * u, src + 32 * DIR * u, n > 32 * u);
}

// Columns [l0, l0 + 16) of M, rows [r0, r1) (all below the block: r0 >= l0 + 16), on
// their way to dst (row i of column l at (l - l0) * ld + i - r0), along M's
// contiguous index, by the warps from FIRST on.
template <int FIRST>
__device__ __forceinline__ void stage(const View& m, int l0, int r0, int r1, float* dst, int ld) {
    constexpr int WARPS = NT / 32 - FIRST;
    const int warp = (int)(threadIdx.x >> 5) - FIRST, lane = threadIdx.x & 31;
    const uint32_t to = (uint32_t)__cvta_generic_to_shared(dst);
    if (warp < 0) return;
    if (m.row_fast) {
        for (int l = warp; l < SB; l += WARPS) {
            const float* src = m.A + (l0 + l) * m.cs + (r0 + lane) * m.rs;
            const uint32_t d = to + 4 * (l * ld + lane);
            if (m.rs > 0) stage_run<1, 32>(src, d, r1 - r0 - lane);
            else stage_run<-1, 32>(src, d, r1 - r0 - lane);
        }
    } else {
        const int l = lane & 15, row = 2 * warp + (lane >> 4);
        const float* src = m.A + (l0 + l) * m.cs + (r0 + row) * m.rs;
        const int64_t step = 2 * WARPS * m.rs;
        uint32_t d = to + 4 * (l * ld + row);
        for (int n = r1 - r0 - row; n > 0; n -= 8 * WARPS, d += 32 * WARPS)
#pragma unroll
            for (int u = 0; u < 4; ++u, src += step)
                cp_async4_if(d + 8 * WARPS * u, src, n > 2 * WARPS * u);
    }
}

// The strictly lower part of the diagonal tile at s0 (column j's rows at 16 j); the
// other words stay as they are and are not used.
__device__ __forceinline__ void stage_tile(const View& m, int s0, float* dst) {
    static_assert(NT == SB * SB, "a thread a word");
    const int a = threadIdx.x & 15, b = threadIdx.x >> 4;
    const int i = m.row_fast ? a : b, j = m.row_fast ? b : a;
    if (i > j && s0 + i < m.k)
        cp_async4((uint32_t)__cvta_generic_to_shared(dst + j * SB + i),
                  m.A + (s0 + i) * m.rs + (s0 + j) * m.cs);
}

// acc += sM(l, i0 .. i0+TR) x(l, 4 columns) over the staged 16 columns; rows in
// packed pairs.
template <int W, int TR>
__device__ __forceinline__ void tile_product(const float* sM, int ld, int i0, const float* x,
                                             uint64_t (&acc)[TR / 2][4]) {
#pragma unroll 4
    for (int l = 0; l < SB; ++l) {
        uint64_t t[TR / 2], b[4];
        const float* mp = sM + l * ld + i0;
        if constexpr (TR >= 4) {
#pragma unroll
            for (int r = 0; r < TR / 4; ++r) {
                const ulonglong2 q = *reinterpret_cast<const ulonglong2*>(mp + 4 * r);
                t[2 * r] = q.x;
                t[2 * r + 1] = q.y;
            }
        } else {
            t[0] = *reinterpret_cast<const uint64_t*>(mp);
        }
        const float4 xv = *reinterpret_cast<const float4*>(x + l * LDC<W>);
        b[0] = pack2(xv.x, xv.x);
        b[1] = pack2(xv.y, xv.y);
        b[2] = pack2(xv.z, xv.z);
        b[3] = pack2(xv.w, xv.w);
#pragma unroll
        for (int r = 0; r < TR / 2; ++r)
#pragma unroll
            for (int v = 0; v < 4; ++v) acc[r][v] = ffma2(t[r], b[v], acc[r][v]);
    }
}

// Rank-16 update of the rows from s0 + 32 on by block s0's; a warp's lanes hold 4
// columns of TR rows each, and the FIRST warps, which come from the next block, take
// their rows last. sM: the block's columns, row s0 + 16 first.
template <int W, int TR, int FIRST>
__device__ __forceinline__ void update(float* sC, const float* sM, int ld, int s0, int k) {
    constexpr int CG = W / 4, RG = 32 / CG;
    constexpr int WARPS = NT / 32;
    const int at = ((threadIdx.x >> 5) + WARPS - FIRST) % WARPS;
    const int lane = threadIdx.x & 31, cg = lane % CG;
    for (int i0 = s0 + 2 * SB + TR * (RG * at + lane / CG); i0 < k; i0 += TR * RG * WARPS) {
        uint64_t acc[TR / 2][4] = {};
        tile_product<W, TR>(sM, ld, i0 - s0 - SB, sC + s0 * LDC<W> + 4 * cg, acc);
#pragma unroll
        for (int r = 0; r < TR / 2; ++r) {
            float lo[4], hi[4];
#pragma unroll
            for (int v = 0; v < 4; ++v) unpack2(acc[r][v], lo[v], hi[v]);
            if (i0 + 2 * r < k) {
                float4* c = reinterpret_cast<float4*>(sC + (i0 + 2 * r) * LDC<W> + 4 * cg);
                const float4 o = *c;
                *c = make_float4(o.x - lo[0], o.y - lo[1], o.z - lo[2], o.w - lo[3]);
            }
            if (i0 + 2 * r + 1 < k) {
                float4* c = reinterpret_cast<float4*>(sC + (i0 + 2 * r + 1) * LDC<W> + 4 * cg);
                const float4 o = *c;
                *c = make_float4(o.x - hi[0], o.y - hi[1], o.z - hi[2], o.w - hi[3]);
            }
        }
    }
}

// Column `c` of the block at s0: its rows less the 16 before them times `cols`
// (row s0's first; not for the first block), then the substitution with `tile`
// (column j's rows at 16 j). Rows past k compute on stale words and are not stored.
template <int W>
__device__ __forceinline__ void solve_block(float* sC, const float* cols, int ld, const float* tile,
                                            const float* sD, int s0, int k, int c) {
    uint64_t x[SB / 2], acc[SB / 2] = {};
    if (s0 > 0) {
#pragma unroll 4
        for (int l = 0; l < SB; ++l) {
            const float v = sC[(s0 - SB + l) * LDC<W> + c];
            const uint64_t b = pack2(v, v);
#pragma unroll
            for (int q = 0; q < SB / 2; q += 2) {
                const ulonglong2 t = *reinterpret_cast<const ulonglong2*>(cols + l * ld + 2 * q);
                acc[q] = ffma2(t.x, b, acc[q]);
                acc[q + 1] = ffma2(t.y, b, acc[q + 1]);
            }
        }
    }
#pragma unroll
    for (int q = 0; q < SB / 2; ++q) {
        float lo, hi;
        unpack2(acc[q], lo, hi);
        x[q] = pack2(sC[(s0 + 2 * q) * LDC<W> + c] - lo, sC[(s0 + 2 * q + 1) * LDC<W> + c] - hi);
    }
#pragma unroll
    for (int p = 0; p < SB / 2; ++p) {                 // rows in pairs
        float lo, hi;
        unpack2(x[p], lo, hi);
        lo *= sD[s0 + 2 * p];
        hi = fmaf(-tile[2 * p * SB + 2 * p + 1], lo, hi) * sD[s0 + 2 * p + 1];
        x[p] = pack2(lo, hi);
        const uint64_t nlo = pack2(-lo, -lo), nhi = pack2(-hi, -hi);
#pragma unroll
        for (int q = p + 1; q < SB / 2; ++q) {
            const float* t = tile + 2 * p * SB + 2 * q;
            x[q] = ffma2(*reinterpret_cast<const uint64_t*>(t), nlo, x[q]);
            x[q] = ffma2(*reinterpret_cast<const uint64_t*>(t + SB), nhi, x[q]);
        }
    }
#pragma unroll
    for (int q = 0; q < SB / 2; ++q) {
        float lo, hi;
        unpack2(x[q], lo, hi);
        if (s0 + 2 * q < k) sC[(s0 + 2 * q) * LDC<W> + c] = lo;
        if (s0 + 2 * q + 1 < k) sC[(s0 + 2 * q + 1) * LDC<W> + c] = hi;
    }
}

// Block s's columns of M below it lie at the low end of the panel space for even s,
// at the high end for odd s: two neighbours are there together as soon as both fit.
// Row stride 4 mod 8 words: the transposed writes of 16 columns meet in two banks.
__device__ __forceinline__ int panel_ld(int rows) { return ((rows + 7) & ~7) + 4; }

// Block 0's columns and the first two tiles, beside the chunk's own load.
__device__ __forceinline__ void trsm_first(const View& m, float* sP, float* sT) {
    stage_tile(m, 0, sT);
    if (SB < m.k) {
        stage<0>(m, 0, SB, m.k, sP, panel_ld(m.k - SB));
        stage_tile(m, SB, sT + SB * SB);
    }
}

// One barrier per block: the first warps finish block s+1 (its update by block s and
// its substitution) while the others update the rows below it; block s+1's columns
// and block s+2's tile arrive meanwhile. sP: `room` floats of panel space.
template <int W>
__device__ __forceinline__ void trsm_chunk(const View& m, float* sC, float* sP, int room, float* sT,
                                           const float* sD) {
    constexpr int FIRST = (W + 31) / 32;               // warps on the next block
    const int k = m.k, tid = threadIdx.x;
    const auto panel = [&](int s0) {
        const int size = SB * panel_ld(k - s0 - SB);
        return (s0 / SB) & 1 ? sP + room - size : sP;
    };
    const auto tile = [&](int s0) { return sT + ((s0 / SB) & 1) * SB * SB; };
    if (tid < W) solve_block<W>(sC, nullptr, 0, tile(0), sD, 0, k, tid);
    __syncthreads();
    for (int s0 = 0; s0 + SB < k; s0 += SB) {
        const int nx = s0 + SB, ld = panel_ld(k - nx);
        const float* cols = panel(s0);
        const bool more = nx + SB < k;
        const bool both = more && SB * (ld + panel_ld(k - nx - SB)) <= room;
        const auto fetch = [&] { stage<FIRST>(m, nx, nx + SB, k, panel(nx), panel_ld(k - nx - SB)); };
        if (more) {
            stage_tile(m, nx + SB, tile(nx + SB));
            if (both) fetch();
            cp_async_commit();
        }
        if (tid < W) solve_block<W>(sC, cols, ld, tile(nx), sD, nx, k, tid);
        // tiles as tall as the rows fill
        constexpr int RG = (NT - 32 * FIRST) / (W / 4);
        const int rows = k - nx - SB;
        if (rows > 4 * RG) update<W, 8, FIRST>(sC, cols, ld, s0, k);
        else if (rows > 2 * RG) update<W, 4, FIRST>(sC, cols, ld, s0, k);
        else update<W, 2, FIRST>(sC, cols, ld, s0, k);
        if (more && !both) {
            __syncthreads();
            fetch();
            cp_async_commit();
        }
        cp_async_wait<0>();
        __syncthreads();
    }
}

// Rows [r0, r1) (at most 256, r0 a multiple of 16) of the product: the 16-column
// blocks below the diagonal one, then every row's own block at once (its columns
// left of the row, in one strip), then alpha (d_i c_i + acc). Two buffers in sM.
template <int W, int TR>
__device__ __forceinline__ void trmm_band(const View& m, float* sC, float* sM, const float* sD,
                                          float alpha, int r0, int r1) {
    constexpr int CG = W / 4, LD = LDB;
    const int tid = threadIdx.x, cg = tid % CG, rg = tid / CG;
    const int i0 = r0 + TR * rg, own = i0 & ~(SB - 1);
    const int last = (r1 - 1) & ~(SB - 1);             // the last row's own block
    uint64_t acc[TR / 2][4] = {};
    // block l0's rows of the band: those below the block
    const auto fetch = [&](int l0, float* dst) {
        if (l0 < last) {
            const int r = max(r0, l0 + SB);
            stage<0>(m, l0, r, r1, dst + r - r0, LD);
        } else {
            for (int e = tid; e < (r1 - r0 + SB - 1) / SB * SB * SB; e += NT) {
                // neighbours along M's contiguous index
                const int i = r0 + (m.row_fast ? e / 256 * 16 + e % 16 : e >> 4);
                const int l = m.row_fast ? (e >> 4) & 15 : e & 15;
                if (i < r1 && l < (i & 15))
                    cp_async4((uint32_t)__cvta_generic_to_shared(dst + l * LD + i - r0),
                              m.A + i * m.rs + ((i & ~15) + l) * m.cs);
            }
        }
        cp_async_commit();
    };
    fetch(0, sM);
    int buf = 0;
    for (int l0 = 0; l0 <= last; l0 += SB, buf ^= 1) {
        const float* cols = sM + buf * SB * LD;
        if (l0 < last) {
            fetch(l0 + SB, sM + (buf ^ 1) * SB * LD);
            cp_async_wait<1>();
        } else {
            cp_async_wait<0>();
        }
        __syncthreads();
        if (l0 < last) {
            if (i0 < r1 && l0 < own)
                tile_product<W, TR>(cols, LD, i0 - r0, sC + l0 * LDC<W> + 4 * cg, acc);
        } else if (i0 < r1) {
            // only l < i takes part (a zero of M times an Inf below the row would be NaN)
            for (int l = own; l < min(i0 + TR, r1) - 1; ++l) {
                const float4 xv = *reinterpret_cast<const float4*>(sC + l * LDC<W> + 4 * cg);
                const float x[4] = {xv.x, xv.y, xv.z, xv.w};
                const float* t = cols + (l - own) * LD + i0 - r0;
#pragma unroll
                for (int r = 0; r < TR / 2; ++r)
#pragma unroll
                    for (int v = 0; v < 4; ++v) {
                        float lo, hi;
                        unpack2(acc[r][v], lo, hi);
                        if (l < i0 + 2 * r) lo = fmaf(t[2 * r], x[v], lo);
                        if (l < i0 + 2 * r + 1) hi = fmaf(t[2 * r + 1], x[v], hi);
                        acc[r][v] = pack2(lo, hi);
                    }
            }
        }
        __syncthreads();
    }
    // (the barrier above: every read of the band's rows is done)
#pragma unroll
    for (int r = 0; r < TR; ++r) {
        const int i = i0 + r;
        if (i >= r1) break;
        float4* c = reinterpret_cast<float4*>(sC + i * LDC<W> + 4 * cg);
        const float4 o = *c;
        const float d = sD[i];
        float s[4];
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            float lo, hi;
            unpack2(acc[r / 2][v], lo, hi);
            s[v] = (r & 1) ? hi : lo;
        }
        *c = make_float4(alpha * fmaf(d, o.x, s[0]), alpha * fmaf(d, o.y, s[1]),
                         alpha * fmaf(d, o.z, s[2]), alpha * fmaf(d, o.w, s[3]));
    }
}

template <int W>
__device__ __forceinline__ void trmm_chunk(const View& m, float* sC, float* sM, const float* sD,
                                           float alpha) {
    constexpr int RG = NT / (W / 4);                   // row groups; a band: at most 256 rows
    constexpr int TALL = W == 16 ? 4 : 8;
    if (m.k > 2 * RG) {
        for (int r0 = (m.k - 1) / (TALL * RG) * (TALL * RG); r0 >= 0; r0 -= TALL * RG)
            trmm_band<W, TALL>(m, sC, sM, sD, alpha, r0, min(m.k, r0 + TALL * RG));
    } else {
        trmm_band<W, 2>(m, sC, sM, sD, alpha, 0, m.k);
    }
}

// Elements of a chunk's column-or-row runs, each by the thread that `copy` gave it.
template <int W, typename F>
__device__ __forceinline__ void each_own(bool row_fast, int k, int nc, F&& f) {
    const int tid = threadIdx.x;
    if (row_fast) {
        for (int c = tid >> 5; c < nc; c += NT / 32)
#pragma unroll 4
            for (int i = tid & 31; i < k; i += 32) f(i, c);
    } else if (tid % W < nc) {
#pragma unroll 4
        for (int i = tid / W; i < k; i += NT / W) f(i, tid % W);
    }
}

// One chunk: `nc` columns of C from column c0 in, through the operation, and out.
// `between` runs once the chunk's loads are on their way.
template <int W, typename F>
__device__ __forceinline__ void chunk(const BatchDesc& d, const View& m, float* sC, float* sT,
                                      const float* sD, int64_t c0, int nc, F&& between) {
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    float* C = static_cast<float*>(d.C) + c0 * d.c_cs;
    const bool row_fast = d.c_rs == 1 || d.c_rs == -1;
    const int rows = (m.k + SB - 1) / SB * SB;         // panel space: what the chunk leaves
    if (d.trsm) trsm_first(m, sC + rows * LDC<W>, sT);
    // a warp a column where the rows are contiguous, else W lanes a row
    const uint32_t to = (uint32_t)__cvta_generic_to_shared(sC);
    if (row_fast) {
        for (int c = warp; c < nc; c += NT / 32) {
            const float* src = C + c * d.c_cs + lane * d.c_rs;
            const uint32_t dst = to + 4 * (lane * LDC<W> + c);
            if (d.c_rs > 0) stage_run<1, 32 * LDC<W>>(src, dst, m.k - lane);
            else stage_run<-1, 32 * LDC<W>>(src, dst, m.k - lane);
        }
    } else if (tid % W < nc) {
        const float* src = C + tid % W * d.c_cs + tid / W * d.c_rs;
        const int64_t step = NT / W * d.c_rs;
        uint32_t dst = to + 4 * (tid / W * LDC<W> + tid % W);
#pragma unroll 4
        for (int n = m.k - tid / W; n > 0; n -= NT / W, src += step, dst += 4 * (NT / W) * LDC<W>)
            cp_async4(dst, src);
    }
    cp_async_commit();
    if (tid % W >= nc)
        for (int i = tid / W; i < m.k; i += NT / W) sC[i * LDC<W> + tid % W] = 0.f;
    between();
    cp_async_wait<0>();
    if (d.trsm && d.alpha != 1.0) {
        const float in = (float)d.alpha;
        each_own<W>(row_fast, m.k, nc, [&](int i, int c) { sC[i * LDC<W> + c] *= in; });
    }
    __syncthreads();
    if (d.trsm) trsm_chunk<W>(m, sC, sC + rows * LDC<W>, SPACE - rows * LDC<W>, sT, sD);
    else trmm_chunk<W>(m, sC, sC + SPACE - 2 * SB * LDB, sD, (float)d.alpha);
    __syncthreads();
    each_own<W>(row_fast, m.k, nc,
                [&](int i, int c) { C[i * d.c_rs + c * d.c_cs] = sC[i * LDC<W> + c]; });
    __syncthreads();
}

// Lines of a matrix of `run` contiguous words (stride `rs`) by `n` such runs toward
// L2: 16 lanes a run. tri: runs of a triangle, from the run's own index on (+1) or up
// to it (-1).
__device__ __forceinline__ void prefetch(const float* p, int run, int64_t rs, int n, int64_t cs,
                                         int tri) {
    for (int f = threadIdx.x >> 4; f < n; f += NT / 16)
        for (int w = (threadIdx.x & 15) * 32; w < run; w += 512)
            if (tri == 0 || (tri > 0 ? w + 32 > f : w <= f))
                asm volatile("prefetch.global.L2 [%0];" ::"l"(p + w * rs + f * cs));
}

__device__ __forceinline__ void prefetch_problem(const BatchDesc& d) {
    if (d.trsm == 2) return;
    const bool mf = d.a_rs == 1 || d.a_rs == -1, cf = d.c_rs == 1 || d.c_rs == -1;
    prefetch(static_cast<const float*>(d.A), (int)d.k, mf ? d.a_rs : d.a_cs, (int)d.k,
             mf ? d.a_cs : d.a_rs, mf ? 1 : -1);
    const int nc = (int)min(d.nrhs, (int64_t)64);
    prefetch(static_cast<const float*>(d.C), cf ? (int)d.k : nc, cf ? d.c_rs : d.c_cs,
             cf ? nc : (int)d.k, cf ? d.c_cs : d.c_rs, 0);
}

// Three problems are on the way at a time: the one at work, the next one, whose
// matrices move toward L2 meanwhile, and the one after it, of which the index and the
// descriptor are being fetched. (Without that a problem of order 16 took 4.5 us, all
// of it a chain of memory latencies.) The last three rounds of problems are taken one
// at a time, so that no CTA holds two while another has none.
__global__ void __launch_bounds__(NT, 2) batched_f32_kernel(const BatchDesc* descs, int64_t count,
                                                            int* counter) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    // chunk: row i, column c at i * LDC + c; M's columns behind it
    float* sC = reinterpret_cast<float*>(smem_raw);
    float* sT = sC + SPACE;                                // two diagonal tiles
    float* sD = sT + 2 * SB * SB;                          // reciprocal (TRSM) or plain diagonal
    __shared__ BatchDesc s_desc[3];
    __shared__ int s_idx[3];
    pdl_trigger();
    pdl_wait();
    const int tid = threadIdx.x;
    // problem blockIdx.x first, the rest in turn; `none`: not taken yet
    const auto take = [&] { return (int)gridDim.x + atomicAdd(counter, 1); };
    constexpr int none = -1;
    const auto early = [&](int idx) { return idx + 3 * (int64_t)gridDim.x < count; };
    if (tid == 0) {
        s_idx[0] = blockIdx.x;
        s_desc[0] = descs[blockIdx.x];
        s_idx[1] = early(blockIdx.x) ? take() : none;
        if (s_idx[1] != none && s_idx[1] < count) s_desc[1] = descs[s_idx[1]];
    }
    __syncthreads();
    prefetch_problem(s_desc[0]);
    for (int at = 0;; at = at == 2 ? 0 : at + 1) {
        if (s_idx[at] == none) {
            __syncthreads();
            if (tid == 0) {
                s_idx[at] = take();
                if (s_idx[at] < count) s_desc[at] = descs[s_idx[at]];
            }
            __syncthreads();
            if (s_idx[at] < count) prefetch_problem(s_desc[at]);
        }
        if (s_idx[at] >= count) break;
        const int nx = at == 2 ? 0 : at + 1, nn = nx == 2 ? 0 : nx + 1;
        int after = none;
        if (tid == 0 && s_idx[nx] != none && early(s_idx[at])) after = take();
        const BatchDesc d = s_desc[at];
        const auto ahead = [&] {
            if (s_idx[nx] != none && s_idx[nx] < count) prefetch_problem(s_desc[nx]);
            if (tid == 0) {
                s_idx[nn] = after;
                if (after != none && after < count) {
                    constexpr int WORDS = sizeof(BatchDesc) / 8;
                    const uint32_t to = (uint32_t)__cvta_generic_to_shared(&s_desc[nn]);
#pragma unroll
                    for (int w = 0; w < WORDS; ++w)
                        asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(to + 8 * w),
                                     "l"(reinterpret_cast<const uint64_t*>(descs + after) + w)
                                     : "memory");
                }
                cp_async_commit();
            }
        };
        const int k = (int)d.k;
        if (d.trsm == 2) {   // alpha == 0: B := 0, A is not read
            ahead();
            float* C = static_cast<float*>(d.C);
            for (int64_t e = tid; e < d.k * d.nrhs; e += NT)
                C[(e % d.k) * d.c_rs + (e / d.k) * d.c_cs] = 0.f;
            cp_async_wait<0>();
            __syncthreads();
            continue;
        }
        const View m{static_cast<const float*>(d.A), d.a_rs, d.a_cs, k,
                     d.a_rs == 1 || d.a_rs == -1};
        for (int i = tid; i < k; i += NT) {
            const float dg = d.unit ? 1.f : m.A[(int64_t)i * (m.rs + m.cs)];
            sD[i] = d.trsm ? 1.f / dg : dg;
        }
        for (int64_t c0 = 0; c0 < d.nrhs;) {
            const int64_t left = d.nrhs - c0;
            const int w = left <= 16 ? 16 : left <= 32 ? 32 : (int)batch_f32_chunk(k);
            const int nc = (int)min((int64_t)w, left);
            const auto between = [&] { if (c0 == 0) ahead(); };
            if (w == 64) chunk<64>(d, m, sC, sT, sD, c0, nc, between);
            else if (w == 32) chunk<32>(d, m, sC, sT, sD, c0, nc, between);
            else chunk<16>(d, m, sC, sT, sD, c0, nc, between);
            c0 += nc;
        }
    }
}

}  // namespace

cudaError_t batched_f32_configure() {
    return cudaFuncSetAttribute(batched_f32_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)SMEM);
}
int batched_f32_ctas_per_sm() {
    int n = 0;
    const cudaError_t e =
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, batched_f32_kernel, NT, SMEM);
    return (e == cudaSuccess && n > 0) ? n : 1;
}
cudaError_t launch_batched_f32(const BatchDesc* descs, int64_t count, int* counter, int grid,
                               cudaStream_t s) {
    return launch_kernel(batched_f32_kernel, dim3(grid), dim3(NT), SMEM, s, descs, count, counter);
}

}  // namespace trx
