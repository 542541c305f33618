// FP32 TRSM with few right-hand sides as one persistent launch on the CUDA
// cores.
//
// With a thin right-hand side the recursion of Section 3.1 is a long chain
// of small launches (a leaf and a GEMM update per 128 rows), each bound by
// latency: at order 8192 with 16 right-hand sides the chain takes about
// 1.4 ms to read a 128 MB triangle. Here the canonical lower M is cut into
// 64-row blocks and the right-hand side into 16-column panels, and task
// (i, p) runs the blocked forward substitution of block row i, left-looking:
//
//     S'   = sum_{j < i-1} M_ij X_jp        (64 x 64 x 16 products, FP32 FMA)
//     P    = inv(M_ii) (alpha B_ip - S')
//     X_ip = P - Z X_i-1,p,   Z = inv(M_ii) M_i,i-1
//
// then writes X_ip into C and publishes it. inv(M_ii) (substitution against
// the identity, FP32, one reciprocal of each diagonal entry: the leaf solve
// of Section 3.3 as a product with the inverted block) and Z are made by
// the task before its first wait when the right-hand side is one panel,
// and by a preparatory pass (thin_prep_kernel, one CTA per block row, the
// same code) when it is several, so the panels' tasks of a block row do not
// each repeat them; the products of a task start as soon as the blocks X_jp
// they need are published, so the reads of M (every element once per
// panel, the dominant traffic) overlap the chain of diagonal blocks; the
// chain itself is one 64 x 64 x 16 product per block.
//
// The same launch also serves as the recursion's leaf for 65 .. 1536
// right-hand sides (the thin leaves): on a leaf's rows, its columns of M
// and its rows of C, with the tensor-core updates between leaves.
//
// A task is eight consecutive block rows of a panel, one a CTA of a cluster. A
// finished block goes to the next four CTAs by st.async into their shared memory
// (with an mbarrier each, 0.2 us), and to everyone as 1024 tagged 64-bit words (FP32
// bits in the low half, 1 in the high half; a 64-bit access is single-copy atomic, so
// value and tag arrive together): a consumer polls the words themselves, one L2
// round trip (0.64 us a poll, 1.5 us from store to use), with no flag and no fence
// between data and signal. The words are zeroed by a memset before each launch.
//
// Four warps of a CTA bring in the tiles of M through a ring of cp.async stages, the
// eight others do the products. Bound by the chain: from X_i-2's arrival a CTA does
// three products (its last tile, the inverse, Z) of 0.5-0.67 us each in two steps.
// us, this kernel against one CTA per ticket that published through L2 only, staged M
// between its products and had a thread on 4 rows x 1 column: 8191 x 16 transposed
// 323 -> 225, 8192 x 16 323 -> 208, 8192 x 64 449 -> 316, a 2048-row leaf with 256
// right-hand sides 121 -> 87. On the way: the products alone 309, clusters with M
// still staged between them 283.
//
// Tasks are taken in order from an atomic counter (block row major), so a
// task only waits for tasks taken before it, which are running or done: the
// solve progresses whatever the number of resident clusters. Every wait is
// bounded: past the budget the CTA writes TRX_ERR_TIMEOUT to the error word
// and the launch's stop word, and every waiting CTA then stops.
//
// Arithmetic: FP32 FMA throughout (no operand split), partial sums in a
// fixed order, so results are bitwise repeatable. A product with the inverted block
// leaves a residual of the size of |M_ii| |inv(M_ii)| |right-hand side|, which an
// ill-conditioned block makes larger than substitution's; such blocks (kMaxGrowth) keep
// M_ii and M_i,i-1 in place of the inverse and Z, and are solved by substitution.
#include <cuda_runtime.h>
#include <stdint.h>

#include "common.cuh"

namespace trx {
namespace thin {

constexpr int BR = kThinBlock;       // rows of a block
constexpr int NP = kThinPanel;       // columns of a panel
constexpr int NT = 256;
constexpr int LD = BR + 4;           // shared row stride (floats): 16-byte aligned rows
constexpr int LDT = BR + 1;          // inverse work tile: conflict-free column reads
constexpr int CL = 8;                // block rows of a task, CTAs of a cluster
constexpr int ND = 4;                // block rows that a CTA pushes its block to
constexpr size_t kAlone = 120 * 1024;   // shared memory that leaves no room for a second CTA
constexpr int NTP = 128;             // threads of the solve that bring in M
constexpr int kTimeout = 4;          // TRX_ERR_TIMEOUT
// Largest |inv(M_ii)| |M_ii| 1 (over rows, in parts of eight columns) of a block that is
// solved by its inverse. Right-hand sides M x of random 64 x 64 triangles, entries below
// the diagonal up to s (diagonal 1 + |N(0,1)|): the componentwise backward error of
// substitution / of the inverse is 4.1e-7 / 1.0e-7 at s = 1/16 (growth 3), 1.9e-7 /
// 2.2e-7 at 1/2 (29), 1.6e-7 / 1.2e-6 at 1 (370).
constexpr float kMaxGrowth = 32.0f;

struct Params {
    int64_t k, nrhs;
    const float* A;
    int64_t a_rs, a_cs;
    float* C;
    int64_t c_rs, c_cs;
    float alpha;
    int unit;
    int nbr, npan;
    int64_t ntask;   // TRMM: tasks in all
    int* ticket;     // next task
    int* stop;       // set by a CTA whose wait ran out: the others stop waiting
    // published blocks: X_ip as 64 x 16 tagged words (FP32 bits, tag 1 in
    // the high half), tile (p, i) at words [(p nbr + i) 1024, + 1024),
    // row-major; zeroed by the launch's memset, so a tag of 1 means "this
    // element of this launch"
    unsigned long long* xt;
    int* err;
    long long wait_ns;
    int withhold;    // test hook: block row 0 is never published (waits run out)
    // inv(M_ii) and Z_i for every block row, made once by thin_prep_kernel
    // when the launch has several panels (block row i at [2 i, 2 i + 2)
    // tiles of BR x LD floats: inv, then Z); nullptr: each task makes its own
    const float* invz;
};

// Ring stages: STAGES - 1 tiles in flight (cp.async); four stages measured
// the same as three.
constexpr int STAGES = 3;

struct Smem {
    // M_ij tiles, k-major: m[s][kk * LD + r] = M[i0 + r][j0 + kk]; tile j of
    // a task's sum sits in stage (j + 1) % STAGES (stage 0 also serves as the
    // work tile of the inverse and of Z before)
    float m[STAGES][BR * LD];
    // inv(M_ii), k-major: inv[kk * LD + r] = Inv[r][kk], and Z = inv(M_ii) M_i,i-1; with
    // inv[BR] != 0 M_ii with its diagonal's reciprocals, and M_i,i-1
    float inv[BR * LD];
    float z[BR * LD];
    float x[2][BR * NP];     // X_jp tiles / right-hand side: x[.][kk * NP + c]
    float near[ND][BR * NP];  // X_i-1 .. X_i-ND as the cluster's CTAs push them
    float dinv[BR];
    unsigned long long near_full[ND];                // mbarriers: `near`,
    unsigned long long full[STAGES], empty[STAGES];  // the stages of m
    int pushed[ND];          // set by the CTA that has sent a block to `near`
    int task;
};
constexpr unsigned long long kTag = 1ull << 32;

__device__ __forceinline__ unsigned long long ld_relaxed64(const unsigned long long* p) {
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.b64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
// two words, each an access of its own to the memory model (16-byte aligned)
__device__ __forceinline__ void st_relaxed64x2(unsigned long long* p, unsigned long long u,
                                               unsigned long long v) {
    asm volatile("st.relaxed.gpu.global.v2.b64 [%0], {%1, %2};" ::"l"(p), "l"(u), "l"(v) : "memory");
}

// barrier of the NT threads that compute
__device__ __forceinline__ void sync_nt() { asm volatile("bar.sync 1, %0;" ::"n"(NT) : "memory"); }
// The same, and whether any of them passed true: the verdict comes with the barrier, so
// that all leave a step together (a flag in shared memory could be set for the next
// step by a fast warp before a slow one has read it for this one).
__device__ __forceinline__ bool sync_nt_any(bool v) {
    uint32_t r;
    asm volatile(
        "{ .reg .pred p, q; setp.ne.u32 q, %1, 0;\n"
        "bar.red.or.pred p, 1, %2, q;\n"
        "selp.u32 %0, 1, 0, p; }"
        : "=r"(r)
        : "r"((uint32_t)v), "n"(NT)
        : "memory");
    return r != 0;
}

__device__ __forceinline__ uint64_t gtimer() {
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}
constexpr int Q = (BR * NP) / NT;    // tagged words of a block per thread

// Issue the loads of this thread's four words of X_jp (all in flight; the
// values are checked by finish_x, so they can be issued a step ahead).
__device__ __forceinline__ void issue_x(const Params& p, int pn, int j,
                                        unsigned long long (&w)[Q]) {
    const unsigned long long* src = p.xt + ((int64_t)pn * p.nbr + j) * (BR * NP) + 2 * threadIdx.x;
#pragma unroll
    for (int q = 0; q < Q; q += 2)
        asm volatile("ld.relaxed.gpu.global.v2.b64 {%0, %1}, [%2];"
                     : "=l"(w[q]), "=l"(w[q + 1])
                     : "l"(src + NT * q)
                     : "memory");
}

// X_jp into `x` from its tagged words: a word loaded before it was
// published (tag 0) is polled again (single-copy atomic 64-bit loads: value
// and tag arrive together), at most wait_ns. False on timeout (the error
// word and the launch's stop word are set) or once another CTA has stopped
// the launch.
__device__ bool finish_x(const Params& p, float* x, int pn, int j,
                         const unsigned long long (&w)[Q]) {
    const unsigned long long* src = p.xt + ((int64_t)pn * p.nbr + j) * (BR * NP);
    const int t = threadIdx.x;
    bool ok = true;
#pragma unroll
    for (int q = 0; q < Q; ++q) {
        const int idx = 2 * t + NT * (q & ~1) + (q & 1);
        unsigned long long v = w[q];
        if (v < kTag) {
            const uint64_t t0 = gtimer();
            while ((v = ld_relaxed64(src + idx)) < kTag) {
                
                if (*(volatile int*)p.stop) { ok = false; break; }
                if (gtimer() - t0 > (uint64_t)p.wait_ns) {
                    atomicExch(p.err, kTimeout);
                    atomicExch(p.stop, 1);
                    ok = false;
                    break;
                }
            }
            if (!ok) break;
        }
        x[idx] = __uint_as_float((unsigned)v);
    }
    return ok;
}

// ---- blocks pushed from one CTA of a cluster to the next ones --------------
__device__ __forceinline__ uint32_t smem_u32(const void* p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ int cluster_rank() {
    int r;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ uint32_t map_rank(uint32_t addr, int rank) {
    uint32_t r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ bool try_wait(uint32_t bar, int parity) {
    uint32_t done;
    asm volatile(
        "{ .reg .pred p; mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n"
        "selp.u32 %0, 1, 0, p; }"
        : "=r"(done)
        : "r"(bar), "r"(parity)
        : "memory");
    return done;
}
// Bounded like finish_x.
__device__ bool wait_bar(const Params& p, const unsigned long long* bar, int parity) {
    const uint32_t a = smem_u32(bar);
    if (try_wait(a, parity)) return true;
    const uint64_t t0 = gtimer();
    while (!try_wait(a, parity)) {
        if (*(volatile int*)p.stop) return false;
        if (gtimer() - t0 > (uint64_t)p.wait_ns) {
            atomicExch(p.err, kTimeout);
            atomicExch(p.stop, 1);
            return false;
        }
    }
    return true;
}
// For a block that is known to be under way.
__device__ void wait_landed(const unsigned long long* bar) {
    const uint64_t t0 = gtimer();
    while (!try_wait(smem_u32(bar), 0) && gtimer() - t0 < 1000000000ull) {}
}
// This thread's two columns of one row of X_i into slot `slot` of CTA `rank`, which
// counts the bytes as they land.
__device__ __forceinline__ void push_near(const Smem& sm, int slot, int rank, int at, float u,
                                          float v) {
    asm volatile(
        "st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v2.b32 [%0], {%1, %2}, [%3];" ::"r"(
            map_rank(smem_u32(&sm.near[slot][at]), rank)),
        "r"(__float_as_uint(u)), "r"(__float_as_uint(v)),
        "r"(map_rank(smem_u32(&sm.near_full[slot]), rank))
        : "memory");
}

// Tile (i0.., j0..) of M into registers, 16 elements a thread, along M's
// contiguous direction; zero outside the strict lower triangle of the order
// (off-diagonal tiles lie below the diagonal: only the order bounds rows).
__device__ __forceinline__ void load_m(const Params& p, int64_t i0, int64_t j0, bool colmajor,
                                       float (&r)[16]) {
    const int t = threadIdx.x;
    const int rr = colmajor ? (t & 63) : (t >> 6), cc = colmajor ? (t >> 6) : (t & 63);
    const float* src = p.A + (i0 + rr) * p.a_rs + (j0 + cc) * p.a_cs;
    const int64_t step = 4 * (colmajor ? p.a_cs : p.a_rs);
    const int64_t rows_left = p.k - (i0 + rr);      // rows of this thread inside the order
#pragma unroll
    for (int q = 0; q < 16; ++q) {
        const bool in = colmajor ? rows_left > 0 : rows_left > 4 * q;
        r[q] = in ? __ldg(src + q * step) : 0.0f;
    }
}
__device__ __forceinline__ void cp_async4(float* dst, const float* src, bool valid) {
    const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(d), "l"(src),
                 "r"(valid ? 4 : 0)
                 : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_async16(float* dst, const float* src) {
    const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(src) : "memory");
}
// all but the newest STAGES - 2 groups complete: the oldest tile in flight has landed
__device__ __forceinline__ void cp_wait_ring() {
    asm volatile("cp.async.wait_group %0;" ::"n"(STAGES - 2) : "memory");
}

// The producer warps' share of tile (i0.., j0..) of M into `dst` by cp.async: in
// 16-byte copies where M's columns are contiguous and aligned, else element by element
// along M's contiguous direction (8.6 clocks a warp, 0.6 us a tile); rows past the
// order are zero-filled (no read).
__device__ __forceinline__ void issue_m(const Params& p, float* dst, int64_t i0, int64_t j0,
                                        bool colmajor, bool wide) {
    const int t = threadIdx.x - NT;
    if (wide && i0 + BR <= p.k) {
        const int rr = 4 * (t & 15), cc = t >> 4;
        const float* src = p.A + (i0 + rr) + (j0 + cc) * p.a_cs;
        float* d = dst + cc * LD + rr;
#pragma unroll
        for (int q = 0; q < BR * BR / 4 / NTP; ++q, src += 8 * p.a_cs) cp_async16(d + 8 * q * LD, src);
        return;
    }
    const int rr = colmajor ? (t & 63) : (t >> 6), cc = colmajor ? (t >> 6) : (t & 63);
    const float* src = p.A + (i0 + rr) * p.a_rs + (j0 + cc) * p.a_cs;
    const int64_t step = 2 * (colmajor ? p.a_cs : p.a_rs);
    const int64_t rows = p.k - (i0 + rr);
    float* d = dst + cc * LD + rr;
    const int dstep = colmajor ? 2 * LD : 2;
#pragma unroll 8
    for (int q = 0; q < BR * BR / NTP; ++q, src += step, d += dstep) {
        const bool in = colmajor ? rows > 0 : rows > 2 * q;
        cp_async4(d, in ? src : p.A, in);
    }
}

// Packed FP32 pairs: fma.rn.f32x2 does two independent round-to-nearest
// FMAs in one instruction (the same results as two fmaf).
__device__ __forceinline__ uint64_t pk2(float a, float b) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ void upk2(uint64_t r, float& a, float& b) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(r));
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
    uint64_t d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}

// The two rows and two columns of a 64 x 16 block that a thread ends up with.
struct Own {
    int row, col;
};
__device__ __forceinline__ Own own_elements() {
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31, kg = (l >> 2) & 3;
    return {32 * (w >> 2) + 4 * (w & 3) + 16 * (l >> 4) + 2 * (kg & 1), 4 * (l & 3) + 2 * (kg >> 1)};
}
// acc[r][c] += sum_kk a[kk][row + r] * x[kk][col + c] for the thread's rows and columns;
// LOWER: a is lower triangular. Four lanes share a 4 x 4 tile, each with every
// fourth kk, and exchange halves of their sums at the end: 32 vector loads and 128
// packed FMAs a thread for 64 kk. (With a thread on 4 rows x 1 column over all kk,
// 128 loads, shared memory set the pace.) A warp's two row tiles
// lie 16 rows apart, so its M words fall into 32 different banks.
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
    uint64_t d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
template <bool LOWER = false>
__device__ __forceinline__ void mma_tile(const float* a, const float* x, float (&acc)[2][2]) {
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31, ct = l & 3, kg = (l >> 2) & 3;
    const int row = 32 * (w >> 2) + 4 * (w & 3) + 16 * (l >> 4);   // the four rows' first
    const int kend = LOWER ? 32 * (w >> 2) + 4 * (w & 3) : BR;
    const float* ap = a + kg * LD + row;
    const float* xp = x + kg * NP + 4 * ct;
    uint64_t s0[4] = {}, s1[4] = {};       // rows 0, 1 and 2, 3 of the tile by column
#pragma unroll 8
    for (int kk = 0; kk < kend; kk += 4) {
        const ulonglong2 m = *reinterpret_cast<const ulonglong2*>(ap + kk * LD);
        const float4 v = *reinterpret_cast<const float4*>(xp + kk * NP);
        const uint64_t b[4] = {pk2(v.x, v.x), pk2(v.y, v.y), pk2(v.z, v.z), pk2(v.w, v.w)};
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            s0[c] = fma2(m.x, b[c], s0[c]);
            s1[c] = fma2(m.y, b[c], s1[c]);
        }
    }
    if constexpr (LOWER) {
        // the warp's two tiles of rows: nothing right of a row takes part (a zero times
        // an Inf there would make a NaN)
        float s[4][4];                     // row, column
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            upk2(s0[c], s[0][c], s[1][c]);
            upk2(s1[c], s[2][c], s[3][c]);
        }
#pragma unroll
        for (int u = 0; u < 5; ++u) {
            const int kk = kend + 4 * u, left = row - kk - kg;   // rows below: r + left >= 0
            const float4 m = *reinterpret_cast<const float4*>(ap + kk * LD);
            const float4 v = *reinterpret_cast<const float4*>(xp + kk * NP);
            const float a[4] = {m.x, m.y, m.z, m.w}, b[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int r = 0; r < 4; ++r)
#pragma unroll
                for (int c = 0; c < 4; ++c)
                    if (r + left >= 0) s[r][c] = fmaf(a[r], b[c], s[r][c]);
        }
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            s0[c] = pk2(s[0][c], s[1][c]);
            s1[c] = pk2(s[2][c], s[3][c]);
        }
    }
    // lanes kg and kg ^ 1 swap row pairs, then kg and kg ^ 2 column pairs
    uint64_t h[4], f[2];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        const uint64_t got = __shfl_xor_sync(0xffffffffu, kg & 1 ? s0[c] : s1[c], 4);
        h[c] = add2(kg & 1 ? s1[c] : s0[c], got);
    }
#pragma unroll
    for (int c = 0; c < 2; ++c) {
        const uint64_t got = __shfl_xor_sync(0xffffffffu, kg & 2 ? h[c] : h[c + 2], 8);
        f[c] = add2(kg & 2 ? h[c + 2] : h[c], got);
        float lo, hi;
        upk2(f[c], lo, hi);
        acc[0][c] += lo;
        acc[1][c] += hi;
    }
}

// inv(M_ii) into sm.inv. M_ii's lower triangle goes to a work tile (aliasing
// sm.m) with rows past the order as identity rows; warp w then solves
// M y = e_c for columns c = 8w .. 8w + 7, lane l holding rows l and l + 32:
// at step r the lane owning row r finishes y_r = (delta_rc - s_r) / m_rr
// (reciprocal of m_rr made once), broadcasts it, and every lane adds
// m_row,r y_r into the partial sums of its later rows. Returns whether the block is to be
// solved by substitution (then M_ii itself is in sm.inv).
__device__ bool invert_diag(const Params& p, Smem& sm, int64_t i0) {
    float* T = sm.m[0];
    float* V = sm.x[0];                                    // |M_ii| 1
    unsigned* growth = reinterpret_cast<unsigned*>(sm.x[1]);
    const int t = threadIdx.x, w = t >> 5, l = t & 31;
    const bool colmajor = p.a_rs == 1 || p.a_rs == -1;
    // all loads in flight at once (one after the other they took most of the time)
    float v[16];
#pragma unroll
    for (int q = 0; q < 16; ++q) {
        const int rr = colmajor ? (t & 63) : (t >> 6) + 4 * q;
        const int cc = colmajor ? (t >> 6) + 4 * q : (t & 63);
        const bool read = i0 + rr < p.k && (cc < rr || (cc == rr && !p.unit));
        v[q] = read ? __ldg(p.A + (i0 + rr) * p.a_rs + (i0 + cc) * p.a_cs) : rr == cc ? 1.0f : 0.0f;
    }
#pragma unroll
    for (int q = 0; q < 16; ++q) {
        const int rr = colmajor ? (t & 63) : (t >> 6) + 4 * q;
        const int cc = colmajor ? (t >> 6) + 4 * q : (t & 63);
        T[rr * LDT + cc] = v[q];
    }
    sync_nt();
    if (t < BR) {
        sm.dinv[t] = 1.0f / T[t * LDT + t];
        float sum = 0.0f;
#pragma unroll 16
        for (int c = 0; c < BR; ++c) sum += fabsf(T[t * LDT + c]);
        V[t] = sum;
    } else if (t == BR) {
        *growth = 0u;
    }
    sync_nt();
    float y0[8], y1[8];          // rows l and l + 32, columns 8 w + u
#pragma unroll
    for (int u = 0; u < 8; ++u) y0[u] = y1[u] = 0.0f;
    // (rows above the warp's columns: zeros)
    for (int r = 8 * w; r < 32; ++r) {           // lane r owns row r
        const float dr = sm.dinv[r];
        const float m0 = T[l * LDT + r], m1 = T[(l + 32) * LDT + r];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const float v = (((r == 8 * w + u) ? 1.0f : 0.0f) - y0[u]) * dr;
            const float yr = __shfl_sync(0xffffffffu, v, r);
            y0[u] = l > r ? fmaf(m0, yr, y0[u]) : l == r ? yr : y0[u];
            y1[u] = fmaf(m1, yr, y1[u]);
        }
    }
    for (int r = w < 4 ? 32 : 8 * w; r < BR; ++r) {   // lane r - 32 owns row r
        const float dr = sm.dinv[r];
        const float m1 = T[(l + 32) * LDT + r];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const float v = (((r == 8 * w + u) ? 1.0f : 0.0f) - y1[u]) * dr;
            const float yr = __shfl_sync(0xffffffffu, v, r - 32);
            y1[u] = l + 32 > r ? fmaf(m1, yr, y1[u]) : l + 32 == r ? yr : y1[u];
        }
    }
    // s_r accumulated with +: the recurrence above keeps s = sum m y and
    // y_r = (delta - s) / m_rr
    float g0 = 0.0f, g1 = 0.0f;
#pragma unroll
    for (int u = 0; u < 8; ++u) {
        sm.inv[(8 * w + u) * LD + l] = y0[u];
        sm.inv[(8 * w + u) * LD + l + 32] = y1[u];
        g0 = fmaf(fabsf(y0[u]), V[8 * w + u], g0);
        g1 = fmaf(fabsf(y1[u]), V[8 * w + u], g1);
    }
    // (bits of numbers that are not negative, or of a NaN: ordered as they are)
    const unsigned g = __reduce_max_sync(0xffffffffu, max(__float_as_uint(g0), __float_as_uint(g1)));
    if (l == 0) atomicMax(growth, g);
    sync_nt();
    const bool subst = *growth > __float_as_uint(kMaxGrowth);
    if (subst)
        for (int e = t; e < BR * BR; e += NT) {
            const int kk = e / BR, r = e % BR;
            sm.inv[kk * LD + r] = r > kk ? T[r * LDT + kk] : r == kk ? sm.dinv[r] : 0.0f;
        }
    if (t == 0) sm.inv[BR] = subst ? 1.0f : 0.0f;
    sync_nt();
    return subst;
}

// Z = inv(M_ii) M_i,i-1 into sm.z (k-major), M_i,i-1 staged row-major in
// sm.m; thread (ty, tx) forms rows 4 ty .. 4 ty + 3, columns tx + 16 u
// (inv is lower: terms q < 8 (warp + 1) only). For a block solved by substitution
// M_i,i-1 itself.
__device__ void make_z(const Params& p, Smem& sm, int64_t i0, bool colmajor, bool subst) {
    float r[16];
    load_m(p, i0, i0 - BR, colmajor, r);
    const int t = threadIdx.x, ty = t >> 4, tx = t & 15;
    if (subst) {
#pragma unroll
        for (int q = 0; q < 16; ++q) {
            const int rr = colmajor ? (t & 63) : (t >> 6) + 4 * q;
            const int cc = colmajor ? (t >> 6) + 4 * q : (t & 63);
            sm.z[cc * LD + rr] = r[q];
        }
        sync_nt();
        return;
    }
#pragma unroll
    for (int q = 0; q < 16; ++q) {
        const int rr = colmajor ? (t & 63) : (t >> 6) + 4 * q;
        const int cc = colmajor ? (t >> 6) + 4 * q : (t & 63);
        sm.m[0][rr * LD + cc] = r[q];
    }
    sync_nt();
    float acc[4][4];
#pragma unroll
    for (int e = 0; e < 4; ++e)
#pragma unroll
        for (int u = 0; u < 4; ++u) acc[e][u] = 0.0f;
    const int qend = 8 * ((t >> 5) + 1);
    for (int q = 0; q < qend; ++q) {
        const float4 iv = *reinterpret_cast<const float4*>(sm.inv + q * LD + 4 * ty);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const float mv = sm.m[0][q * LD + tx + 16 * u];
            acc[0][u] = fmaf(iv.x, mv, acc[0][u]);
            acc[1][u] = fmaf(iv.y, mv, acc[1][u]);
            acc[2][u] = fmaf(iv.z, mv, acc[2][u]);
            acc[3][u] = fmaf(iv.w, mv, acc[3][u]);
        }
    }
#pragma unroll
    for (int e = 0; e < 4; ++e)
#pragma unroll
        for (int u = 0; u < 4; ++u) sm.z[(tx + 16 * u) * LD + 4 * ty + e] = acc[e][u];
    sync_nt();
}

// rhs := inv(M_ii) rhs by substitution, M_ii in sm.inv as above; a warp two columns, a
// lane rows l and l + 32.
__device__ __noinline__ void substitute(const Smem& sm, float* rhs) {
    const int l = threadIdx.x & 31, c0 = 2 * (threadIdx.x >> 5);
    float v0[2], v1[2];
#pragma unroll
    for (int c = 0; c < 2; ++c) {
        v0[c] = rhs[l * NP + c0 + c];
        v1[c] = rhs[(l + 32) * NP + c0 + c];
    }
#pragma unroll 4
    for (int r = 0; r < 32; ++r) {
        const float d = sm.inv[r * LD + r], m0 = sm.inv[r * LD + l], m1 = sm.inv[r * LD + l + 32];
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            const float x = __shfl_sync(0xffffffffu, v0[c], r) * d;
            v0[c] = l > r ? fmaf(-m0, x, v0[c]) : l == r ? x : v0[c];
            v1[c] = fmaf(-m1, x, v1[c]);
        }
    }
#pragma unroll 4
    for (int r = 32; r < BR; ++r) {
        const float d = sm.inv[r * LD + r], m1 = sm.inv[r * LD + l + 32];
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            const float x = __shfl_sync(0xffffffffu, v1[c], r - 32) * d;
            v1[c] = l + 32 > r ? fmaf(-m1, x, v1[c]) : l + 32 == r ? x : v1[c];
        }
    }
#pragma unroll
    for (int c = 0; c < 2; ++c) {
        rhs[l * NP + c0 + c] = v0[c];
        rhs[(l + 32) * NP + c0 + c] = v1[c];
    }
}

// inv(M_ii) and Z_i = inv(M_ii) M_i,i-1 of block row blockIdx.x into
// p.invz, by the same code (so the same values) as a task of the solve
// makes them; with several panels every task of a block row would repeat it.
__global__ void __launch_bounds__(NT) thin_prep_kernel(const Params p, float* invz) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    Smem& sm = *reinterpret_cast<Smem*>(smem_raw);
    const int i = blockIdx.x;
    const int64_t i0 = (int64_t)i * BR;
    const bool subst = invert_diag(p, sm, i0);
    if (i > 0) make_z(p, sm, i0, p.a_rs == 1 || p.a_rs == -1, subst);
    float4* dst = reinterpret_cast<float4*>(invz + (size_t)i * 2 * BR * LD);
    for (int e = threadIdx.x; e < BR * LD / 4; e += NT) {
        dst[e] = reinterpret_cast<const float4*>(sm.inv)[e];
        if (i > 0) dst[BR * LD / 4 + e] = reinterpret_cast<const float4*>(sm.z)[e];
    }
}

__global__ void __cluster_dims__(CL, 1, 1) __launch_bounds__(NT + NTP, 2)
    thin_trsm_kernel(const Params p) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    Smem& sm = *reinterpret_cast<Smem*>(smem_raw);
    const int t = threadIdx.x;
    const Own own = own_elements();
    const bool colmajor = p.a_rs == 1 || p.a_rs == -1;
    // one task a cluster, in the order of the tickets: CL consecutive block rows of a
    // panel, one a CTA
    const int rank = cluster_rank();
    if (t == 0) {
        for (int q = 0; q < ND; ++q) {
            sm.pushed[q] = 0;
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&sm.near_full[q])));
            asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(
                             smem_u32(&sm.near_full[q])),
                         "r"((int)(BR * NP * sizeof(float)))
                         : "memory");
        }
        for (int q = 0; q < STAGES; ++q) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(&sm.full[q])),
                         "n"(NTP));
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(&sm.empty[q])),
                         "n"(NT / 32));
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        if (rank == 0) sm.task = atomicAdd(p.ticket, 1);
    }
    cluster_sync();
    int task;
    asm volatile("ld.shared::cluster.s32 %0, [%1];"
                 : "=r"(task)
                 : "r"(map_rank(smem_u32(&sm.task), 0)));
    const int i = task / p.npan * CL + rank, pn = task % p.npan;
    const int64_t i0 = (int64_t)i * BR, c0 = (int64_t)pn * NP;
    const int jz = i - 1;                             // blocks j < jz of M go into S'
    if (t >= NT) {
        // producers: tile j of M into stage (j + 1) % STAGES as the stage comes free
        const bool wide = p.a_rs == 1 && p.a_cs % 4 == 0 && ((uintptr_t)p.A & 15) == 0;
        if (i < p.nbr)
            for (int j = 0; j < jz; ++j) {
                const int s = (j + 1) % STAGES, n = j / STAGES;
                if ((s == 0 || n > 0) && !wait_bar(p, &sm.empty[s], (s == 0 ? n : n - 1) & 1)) break;
                issue_m(p, sm.m[s], i0, (int64_t)j * BR, colmajor, wide);
                asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(
                                 smem_u32(&sm.full[s]))
                             : "memory");
            }
    } else while (i < p.nbr) {   // left by the breaks
        // this task's right-hand side rows, read before anything is written
        float b[2][2];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int64_t gi = i0 + own.row + (e & 1), gj = c0 + own.col + (e >> 1);
            b[e & 1][e >> 1] = (gi < p.k && gj < p.nrhs) ? __ldcg(p.C + gi * p.c_rs + gj * p.c_cs) : 0.0f;
        }
        // S' = sum_{j < i-1} M_ij X_jp (X_i-1,p enters through Z), X_jp's words loaded
        // one step ahead
        float acc[2][2] = {};
        unsigned long long w[Q];
        if (p.invz) {
            // inv(M_ii) and Z_i made by thin_prep_kernel
            const float* src = p.invz + (size_t)i * 2 * BR * LD;
            for (int e = t; e < BR * LD / 4; e += NT) {
                cp_async16(sm.inv + 4 * e, src + 4 * e);
                if (i > 0) cp_async16(sm.z + 4 * e, src + BR * LD + 4 * e);
            }
            cp_commit();
        } else {
            const bool subst = invert_diag(p, sm, i0);
            if (i > 0) make_z(p, sm, i0, colmajor, subst);
        }
        const auto release = [&](int s) {
            __syncwarp();
            if (t % 32 == 0)
                asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&sm.empty[s]))
                             : "memory");
        };
        release(0);
        // the nearest blocks are pushed here by the CTAs before this one in the
        // cluster, X_j into slot i - 1 - j; blocks j < far come from xt
        const int far = min(jz, i - min(rank, ND));
        if (far > 0) issue_x(p, pn, 0, w);
        bool stop = false;
        for (int j = 0; j < jz; ++j) {
            const int s = (j + 1) % STAGES;
            const bool ok = (j < far ? finish_x(p, sm.x[j & 1], pn, j, w)
                                     : wait_bar(p, &sm.near_full[i - 1 - j], 0)) &&
                            wait_bar(p, &sm.full[s], j / STAGES & 1);
            if ((stop = sync_nt_any(!ok))) break;   // also: X_j-1 is done with
            if (j + 1 < far) issue_x(p, pn, j + 1, w);
            mma_tile(sm.m[s], j < far ? sm.x[j & 1] : sm.near[i - 1 - j], acc);
            release(s);
        }
        if (stop) break;
        if (i > 0 && rank == 0) issue_x(p, pn, i - 1, w);
        // P = inv(M_ii) (alpha B - S'), then X = P - Z X_i-1,p
        float* rhs = sm.x[(i + 1) & 1];   // the last product (j = i - 2) reads the other
#pragma unroll
        for (int e = 0; e < 4; ++e)
            rhs[(own.row + (e & 1)) * NP + own.col + (e >> 1)] =
                fmaf(p.alpha, b[e & 1][e >> 1], -acc[e & 1][e >> 1]);
        if (p.invz) asm volatile("cp.async.wait_group 0;" ::: "memory");
        sync_nt();
        const bool subst = sm.inv[BR] != 0.0f;
        float xo[2][2] = {};
        if (!subst) mma_tile<true>(sm.inv, rhs, xo);
        if (i > 0) {
            float* prev = sm.x[i & 1];
            const bool ok = rank == 0 ? finish_x(p, prev, pn, i - 1, w)
                                      : wait_bar(p, &sm.near_full[0], 0);
            if (sync_nt_any(!ok)) break;
            float zx[2][2] = {};
            mma_tile(sm.z, rank == 0 ? prev : sm.near[0], zx);
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                if (subst) rhs[(own.row + (e & 1)) * NP + own.col + (e >> 1)] -= zx[e & 1][e >> 1];
                else xo[e & 1][e >> 1] -= zx[e & 1][e >> 1];
            }
        }
        if (subst) {
            sync_nt();
            substitute(sm, rhs);
            sync_nt();
#pragma unroll
            for (int e = 0; e < 4; ++e)
                xo[e & 1][e >> 1] = rhs[(own.row + (e & 1)) * NP + own.col + (e >> 1)];
        }
        // publish the block (tagged words: the chain), then the result in C
        unsigned long long* dst = p.xt + ((int64_t)pn * p.nbr + i) * (BR * NP);
        if (!(p.withhold && i == 0)) {
#pragma unroll
            for (int d = 1; d <= ND; ++d)
                if (rank + d < CL && i + d < p.nbr) {
#pragma unroll
                    for (int r = 0; r < 2; ++r)
                        push_near(sm, d - 1, rank + d, (own.row + r) * NP + own.col, xo[r][0],
                                  xo[r][1]);
                    if (t == 0)
                        asm volatile("st.shared::cluster.s32 [%0], 1;" ::"r"(
                                         map_rank(smem_u32(&sm.pushed[d - 1]), rank + d))
                                     : "memory");
                }
#pragma unroll
            for (int r = 0; r < 2; ++r)
                st_relaxed64x2(dst + (own.row + r) * NP + own.col, kTag | __float_as_uint(xo[r][0]),
                               kTag | __float_as_uint(xo[r][1]));
        }
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int64_t gi = i0 + own.row + (e & 1), gj = c0 + own.col + (e >> 1);
            if (gi < p.k && gj < p.nrhs) p.C[gi * p.c_rs + gj * p.c_cs] = xo[e & 1][e >> 1];
        }
        break;
    }
    // nothing in flight at exit (the producers' copies belong to no group)
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncwarp();
    // no CTA leaves while another may read its task or push to it, nor (after a
    // timeout) before what was pushed has landed
    cluster_sync();
    if (t == 0)
        for (int q = 0; q < ND; ++q)
            if (*(volatile int*)&sm.pushed[q]) wait_landed(&sm.near_full[q]);
}

// ---- TRMM with few right-hand sides ---------------------------------------
// C := alpha M C (canonical lower), one persistent launch after a packing
// pass: task (i, p) forms the 64 x 16 block
//     alpha (sum_{j < i} M_ij B_jp + tril(M_ii) B_ip)
// from a packed copy of C's original rows (so no task reads a block another
// task has overwritten) and writes it into C. The tasks need nothing from
// one another; they are taken longest first (block rows from the bottom),
// M tiles and packed B tiles through a cp.async ring.

struct SmemM {
    float m[STAGES][BR * LD];        // M_ij, k-major (as the TRSM's)
    float x[STAGES][BR * NP];        // packed B_jp tiles, row-major
    float d[BR * LD];                // M_ii's lower triangle (unit: diagonal 1), k-major
    int task;
    int last;                        // this CTA's piece arrived last in its row
};

// C's original rows as tiles: tile (p, j) at Bp[(p nbr + j) * BR * NP],
// element (kk, c) at kk * NP + c; zero past the order and the columns.
__global__ void __launch_bounds__(256) thin_pack_kernel(const Params p, float* Bp) {
    const int64_t e = (int64_t)blockIdx.x * 256 + threadIdx.x;
    const int64_t total = (int64_t)p.npan * p.nbr * (BR * NP);
    if (e >= total) return;
    const int c = (int)(e % NP), kk = (int)((e / NP) % BR);
    const int64_t tile = e / (BR * NP), j = tile % p.nbr, pn = tile / p.nbr;
    const int64_t gi = j * BR + kk, gj = pn * NP + c;
    Bp[e] = (gi < p.k && gj < p.nrhs) ? p.C[gi * p.c_rs + gj * p.c_cs] : 0.0f;
}

// M_ij and B_jp into ring stage s (one commit group).
__device__ __forceinline__ void issue_mb(const Params& p, SmemM& sm, int s, int64_t i0, int j,
                                         const float* btiles, bool colmajor) {
    const int t = threadIdx.x;
    const int rr0 = colmajor ? (t & 63) : (t >> 6), cc0 = colmajor ? (t >> 6) : (t & 63);
    const float* src = p.A + (i0 + rr0) * p.a_rs + ((int64_t)j * BR + cc0) * p.a_cs;
    const int64_t step = 4 * (colmajor ? p.a_cs : p.a_rs);
    const int64_t rows_left = p.k - (i0 + rr0);
#pragma unroll
    for (int q = 0; q < 16; ++q) {
        const int rr = colmajor ? rr0 : rr0 + 4 * q, cc = colmajor ? cc0 + 4 * q : cc0;
        const bool in = colmajor ? rows_left > 0 : rows_left > 4 * q;
        cp_async4(sm.m[s] + cc * LD + rr, in ? src + q * step : p.A, in);
    }
    cp_async16(sm.x[s] + 4 * t, btiles + (int64_t)j * (BR * NP) + 4 * t);   // 256 x 16 B
    cp_commit();
}

// Long block rows are cut into pieces of at most kPiece off-diagonal tiles
// (the last piece also takes the diagonal block), so no task streams more
// than kPiece + 1 tiles; a row of several pieces writes their partial sums
// to slots, and the piece that arrives last (an atomic count per row)
// adds them in piece order, so the result does not depend on which CTA
// finishes when. Pieces of row i: P_i = max(1, ceil(i / kPiece)).
constexpr int kPiece = 32;
__host__ __device__ __forceinline__ int64_t pieces_of(int64_t i) {
    return i == 0 ? 1 : (i + kPiece - 1) / kPiece;
}
// pieces of rows 0 .. r (r >= -1)
__host__ __device__ __forceinline__ int64_t pieces_upto(int64_t r) {
    if (r < 0) return 0;
    const int64_t a = r / kPiece, b = r % kPiece;
    return 1 + (int64_t)kPiece / 2 * a * (a + 1) + b * (a + 1);
}

__global__ void __launch_bounds__(NT, 2) thin_trmm_kernel(const Params p, const float* Bp,
                                                          float* part, int* count) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    SmemM& sm = *reinterpret_cast<SmemM*>(smem_raw);
    const int t = threadIdx.x;
    const Own own = own_elements();
    const bool colmajor = p.a_rs == 1 || p.a_rs == -1;
    const int64_t total = pieces_upto(p.nbr - 1);
    while (true) {
        __syncthreads();
        if (t == 0) sm.task = atomicAdd(p.ticket, 1);
        __syncthreads();
        const int64_t task = sm.task;
        if (task >= p.ntask) break;
        // pieces are taken from the bottom row up: piece index tp counts
        // down from the last row's pieces
        const int64_t tp = task / p.npan;
        const int pn = (int)(task % p.npan);
        int lo = 0, hi = p.nbr - 1;                  // largest i with pieces of rows >= i > tp
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (total - pieces_upto(mid - 1) > tp) lo = mid; else hi = mid - 1;
        }
        const int i = lo;
        const int64_t np_i = pieces_of(i);
        const int q = (int)(tp - (total - pieces_upto(i)));
        const bool last_piece = q == np_i - 1;
        const int jb = q * kPiece, je = (int)((q + 1) * kPiece < i ? (q + 1) * kPiece : i);
        const int64_t i0 = (int64_t)i * BR, c0 = (int64_t)pn * NP;
        const float* btiles = Bp + (int64_t)pn * p.nbr * (BR * NP);
#pragma unroll
        for (int q = 0; q < STAGES - 1; ++q) {      // tiles jb .. jb + STAGES - 2
            if (jb + q < je) issue_mb(p, sm, (jb + q) % STAGES, i0, jb + q, btiles, colmajor);
            else cp_commit();
        }
        if (last_piece) {
            // M_ii's lower triangle, k-major: d[kk][r] = M(r, kk) for kk <= r
            for (int e = t; e < BR * BR; e += NT) {
                const int rr = colmajor ? e % BR : e / BR, cc = colmajor ? e / BR : e % BR;
                const int64_t gi = i0 + rr, gj = i0 + cc;
                float v = 0.0f;
                if (gi < p.k) {
                    if (cc < rr) v = __ldg(p.A + gi * p.a_rs + gj * p.a_cs);
                    else if (cc == rr) v = p.unit ? 1.0f : __ldg(p.A + gi * p.a_rs + gj * p.a_cs);
                }
                sm.d[cc * LD + rr] = v;
            }
        }
        float acc[2][2] = {};
        for (int j = jb; j < je; ++j) {
            cp_wait_ring();                          // this thread's copies of tile j
            __syncthreads();
            // tile j - 1's stage is free: tile j + STAGES - 1 goes there
            if (j + STAGES - 1 < je)
                issue_mb(p, sm, (j + STAGES - 1) % STAGES, i0, j + STAGES - 1, btiles, colmajor);
            else cp_commit();
            mma_tile(sm.m[j % STAGES], sm.x[j % STAGES], acc);
            __syncthreads();
        }
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncthreads();
        if (last_piece) {
            // the diagonal block with B_ip (plain loads into stage 0's x)
            *reinterpret_cast<float4*>(sm.x[0] + 4 * t) =
                *reinterpret_cast<const float4*>(btiles + (int64_t)i * (BR * NP) + 4 * t);
            __syncthreads();
            mma_tile<true>(sm.d, sm.x[0], acc);
        }
        if (np_i > 1) {
            // partial sums to this piece's slot; the last to arrive combines
            float* slots = part + ((int64_t)pn * total + pieces_upto(i - 1)) * (BR * NP);
#pragma unroll
            for (int e = 0; e < 4; ++e)
                __stcg(slots + q * (BR * NP) + (own.row + (e & 1)) * NP + own.col + (e >> 1),
                       acc[e & 1][e >> 1]);
            __threadfence();
            __syncthreads();
            if (t == 0) sm.last = atomicAdd(count + (int64_t)pn * p.nbr + i, 1) == np_i - 1;
            __syncthreads();
            if (!sm.last) continue;
            __threadfence();
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                float sum = 0.0f;
                for (int64_t r = 0; r < np_i; ++r)
                    sum += __ldcg(slots + r * (BR * NP) + (own.row + (e & 1)) * NP + own.col + (e >> 1));
                acc[e & 1][e >> 1] = sum;
            }
        }
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int64_t gi = i0 + own.row + (e & 1), gj = c0 + own.col + (e >> 1);
            if (gi < p.k && gj < p.nrhs) p.C[gi * p.c_rs + gj * p.c_cs] = p.alpha * acc[e & 1][e >> 1];
        }
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
}

}  // namespace thin

// The thin TRSM's scratch: ticket and stop word (16 bytes), the tagged
// words of every (block, panel); with several panels also the block rows' inv / Z
// tiles.
static size_t thin_words_bytes(int64_t nbr, int64_t npan) {
    return 16 + (size_t)(nbr * npan) * kThinBlock * kThinPanel * 8;
}
size_t thin_prep_bytes(int64_t k) {
    return (size_t)((k + kThinBlock - 1) / kThinBlock) * 2 * thin::BR * thin::LD * sizeof(float);
}
size_t thin_scratch_bytes(int64_t k, int64_t nrhs) {
    const int64_t nbr = (k + kThinBlock - 1) / kThinBlock;
    const int64_t npan = (nrhs + kThinPanel - 1) / kThinPanel;
    return thin_words_bytes(nbr, npan) + (npan > 1 ? thin_prep_bytes(k) : 0);
}

// Two clusters fit the same SMs, where each would stage M at half the rate: from
// kSpreadRows block rows on, launches that leave a few SMs over (16 of 19 taken: 128 CTAs
// on 152 SMs, whose parts do not divide into clusters of eight evenly) ask for more shared
// memory than two have room for. us,
// without / with: 8191 x 16 transposed 281 / 230, 8192 x 16 228 / 208, 4096 x 32 131 /
// 117, 2048 x 64 73 / 69, 4096 x 16 115 / 114; but 1024 x 128 48 / 54, 512 x 256 36 / 46
// (the SMs change their split of shared memory between the launches of a call).
constexpr int64_t kSpreadRows = 32;
static int g_thin_trmm_ctas_per_sm = 0;

cudaError_t thin_configure() {
    cudaError_t e0 = cudaFuncSetAttribute(thin::thin_trmm_kernel,
                                          cudaFuncAttributeMaxDynamicSharedMemorySize,
                                          (int)sizeof(thin::SmemM));
    if (e0 != cudaSuccess) return e0;
    int nm = 0;
    e0 = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nm, thin::thin_trmm_kernel, thin::NT,
                                                       sizeof(thin::SmemM));
    if (e0 != cudaSuccess) return e0;
    g_thin_trmm_ctas_per_sm = nm > 0 ? nm : 1;
    cudaError_t e = cudaFuncSetAttribute(thin::thin_trsm_kernel,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)thin::kAlone);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(thin::thin_prep_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)sizeof(thin::Smem));
    if (e != cudaSuccess) return e;
    return cudaSuccess;
}

static thin::Params thin_params(const Canon<float>& c, float alpha) {
    thin::Params p{};
    p.k = c.k;
    p.nrhs = c.nrhs;
    p.A = c.A;
    p.a_rs = c.a_rs;
    p.a_cs = c.a_cs;
    p.C = c.C;
    p.c_rs = c.c_rs;
    p.c_cs = c.c_cs;
    p.alpha = alpha;
    p.unit = c.unit ? 1 : 0;
    p.nbr = (int)((c.k + kThinBlock - 1) / kThinBlock);
    p.npan = (int)((c.nrhs + kThinPanel - 1) / kThinPanel);
    return p;
}

cudaError_t launch_thin_prep(const Canon<float>& c, float* invz, cudaStream_t s) {
    const thin::Params p = thin_params(c, 1.0f);
    thin::thin_prep_kernel<<<(unsigned)p.nbr, thin::NT, sizeof(thin::Smem), s>>>(p, invz);
    return cudaGetLastError();
}

cudaError_t launch_thin_trsm(const Canon<float>& c, float alpha, int* scratch, const float* invz,
                             bool made, int* err, long long wait_ns, int num_sms,
                             cudaStream_t s, bool withhold) {
    if (c.k <= 0 || c.nrhs <= 0) return cudaSuccess;
    const int64_t nbr = (c.k + kThinBlock - 1) / kThinBlock;
    const int64_t npan = (c.nrhs + kThinPanel - 1) / kThinPanel;
    if (nbr * npan > (int64_t)1 << 30) return cudaErrorInvalidValue;
    thin::Params p = thin_params(c, alpha);
    p.ticket = scratch;
    p.stop = scratch + 1;
    p.xt = reinterpret_cast<unsigned long long*>(reinterpret_cast<char*>(scratch) + 16);
    p.err = err;
    p.wait_ns = wait_ns;
    p.withhold = withhold ? 1 : 0;
    // the words (and ticket) are zeroed every launch; inv / Z are written
    cudaError_t e = cudaMemsetAsync(scratch, 0, thin_words_bytes(nbr, npan), s);
    if (e != cudaSuccess) return e;
    if (npan > 1 && invz == nullptr) {
        float* own = reinterpret_cast<float*>(reinterpret_cast<char*>(scratch) +
                                              thin_words_bytes(nbr, npan));
        if (!made && (e = launch_thin_prep(c, own, s)) != cudaSuccess) return e;
        invz = own;
    }
    p.invz = invz;
    const int64_t clusters = (nbr + thin::CL - 1) / thin::CL * npan;
    // a long chain on few enough CTAs for an SM each: shared memory for one
    const bool spread = nbr >= kSpreadRows && clusters * thin::CL * 19 <= (int64_t)num_sms * 16;
    const size_t smem = spread ? thin::kAlone : sizeof(thin::Smem);
    thin::thin_trsm_kernel<<<(unsigned)(clusters * thin::CL), thin::NT + thin::NTP, smem, s>>>(p);
    return cudaGetLastError();
}

// The thin TRMM's scratch: ticket (16 bytes), per-row piece counts, C's
// rows packed by tiles, the pieces' partial sums; zeroed / written by the
// launch itself.
static int64_t align_words(int64_t n) { return (n + 3) / 4 * 4; }   // 16-byte steps (4-byte words)

size_t thin_trmm_scratch_bytes(int64_t k, int64_t nrhs) {
    const int64_t nbr = (k + kThinBlock - 1) / kThinBlock;
    const int64_t npan = (nrhs + kThinPanel - 1) / kThinPanel;
    const int64_t tile = (int64_t)kThinBlock * kThinPanel;
    return 4 * (size_t)(4 + align_words(nbr * npan) + nbr * npan * tile +
                        thin::pieces_upto(nbr - 1) * npan * tile);
}

cudaError_t launch_thin_trmm(const Canon<float>& c, float alpha, int* scratch, int num_sms,
                             cudaStream_t s) {
    if (c.k <= 0 || c.nrhs <= 0) return cudaSuccess;
    const int64_t nbr = (c.k + kThinBlock - 1) / kThinBlock;
    const int64_t npan = (c.nrhs + kThinPanel - 1) / kThinPanel;
    const int64_t total = thin::pieces_upto(nbr - 1);
    if (total * npan > (int64_t)1 << 30) return cudaErrorInvalidValue;
    thin::Params p = thin_params(c, alpha);
    p.ntask = total * npan;
    p.ticket = scratch;
    int* count = scratch + 4;
    float* Bp = reinterpret_cast<float*>(scratch + 4 + align_words(nbr * npan));
    float* part = Bp + nbr * npan * (int64_t)(kThinBlock * kThinPanel);
    cudaError_t e = cudaMemsetAsync(scratch, 0, 4 * (size_t)(4 + align_words(nbr * npan)), s);
    if (e != cudaSuccess) return e;
    const int64_t packed = nbr * npan * (kThinBlock * kThinPanel);
    thin::thin_pack_kernel<<<(unsigned)((packed + 255) / 256), 256, 0, s>>>(p, Bp);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    const int per_sm = g_thin_trmm_ctas_per_sm > 0 ? g_thin_trmm_ctas_per_sm : 1;
    const int64_t cap = (int64_t)num_sms * per_sm;
    const int grid = (int)(p.ntask < cap ? p.ntask : cap);
    thin::thin_trmm_kernel<<<grid, thin::NT, sizeof(thin::SmemM), s>>>(p, Bp, part, count);
    return cudaGetLastError();
}

}  // namespace trx
