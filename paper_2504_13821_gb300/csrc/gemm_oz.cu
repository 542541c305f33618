// FP64 GEMM update on the BF16 tensor cores (tcgen05 + TMEM + bulk copies,
// sm_103a), by the error-free splitting of Ozaki, Ogita, Oishi and Rump
// ("Error-free transformations of matrix multiplication by using fast
// routines of matrix multiplication", Numer. Algorithms 59, 2012):
//
//   C[rc+i, j] = beta * C[rc+i, j] + gamma * sum_l M(rc+i, rk+l) * C[rk+l, j]
//
// the off-diagonal step of the recursion of Section 3.1 in FP64. The FP64 pipe
// of this part does 1.06 TFLOP/s (DFMA probe), the BF16 tensor pipe about
// 1900: 36 BF16 products in place of one FP64 product still leave 47 TFLOP/s.
//
// Arithmetic. Each row r of either operand is scaled by a power of two to
// below 1/2 in magnitude and rounded to a 64-bit fixed-point number, whose
// eight balanced base-256 digits d_1 .. d_8 (weights 2^-8 .. 2^-64, each in
// [-128, 128]) are exact in BF16. The products of digits i and j with
// i + j <= 9 are summed on the tensor cores, one FP32 accumulator per weight
// 2^-8(i+j) ("level" 2 .. 9). A sum of at most 128 * 8 products of two digits
// stays within 2^24, so K chunks of 128 make every level an exact integer;
// chunks are added up exactly in 64-bit integers (levels 2-6) and in FP32
// values of two digits (levels 7-8, level 9 rounded to 2^-64). Left out: the
// digit products of weight below 2^-72. In units of the scaled operands the
// whole sum's error is below K' 2^-62, K' the smaller count of non-zeros of
// the two rows.
//
// When it applies. That error is relative to the rows' largest entries, not
// to sum |m||c| as an FMA chain's is. So the kernel also forms P = |M||C| (one
// BF16 product of the rounded-down magnitudes, 3 % more work) and keeps the
// result of a 32-row x BN/2-column piece only where P >= K' 2^-12 for every
// element, i.e. where its error is below 4 u sum |m||c| (u = 2^-53; the bound
// of a K-term FMA chain is K u sum |m||c|, K >= 64). Pieces that fail, or that
// hold an Inf, a NaN or a row outside 2^+-300, are left as they were and
// flagged, and the DFMA kernel (gemm_simt.cu), launched after this one over
// the flagged pieces only, computes them.
//
// Measured, 2048 x 4096 with K 2048 (operand split, product and the empty DFMA
// pass together): 1002 us, 34 TFLOP/s, against 28519 us by DFMA; 4096^3 41
// TFLOP/s. Relative error against quad precision 5.6e-17 (DFMA 7.7e-16).
#include <stdint.h>

#include "common.cuh"
#include "tc_ptx.cuh"

namespace trx {
namespace oz {

constexpr int S = 8;                         // digits per operand
constexpr int BM = 128;                      // rows of a tile (TMEM lanes)
constexpr int KS = 16;                       // K of one step (one tcgen05.mma)
constexpr int CHUNK = 8;                     // steps per exact sum (128 terms)
constexpr int STAGES = 4;                    // ring depth, one step per stage
constexpr int NT = 320;                      // producer, MMA issuer, 8 epilogue warps
constexpr int kTimeout = 4;                  // TRX_ERR_TIMEOUT
constexpr int kBadExp = 1 << 20;             // row with an Inf, a NaN or out of range
constexpr int kMaxExp = 300;

// Operand image: for each block of BR rows and each K step, S digit planes of
// BR x 16 BF16 in the tensor core's unswizzled K-major layout (8 x 16-byte
// core matrices; the two of a K step side by side), so that a ring stage is
// one contiguous copy per operand and needs no tensor map. The magnitude
// image is the same with a single plane.
__host__ __device__ constexpr int64_t plane_bytes(int br) { return (int64_t)br * KS * 2; }
__device__ __forceinline__ int64_t row_offset(int r) { return (r >> 3) * 256 + (r & 7) * 16; }

struct Operand {                             // element (r, l) = X[r * rs + l * ls]
    const double* X;
    int64_t rs, ls, rows;
    int br;                                  // rows per block
    unsigned char* digits;                   // [block][step][digit][br x 16]
    unsigned char* mags;                     // [block][step][br x 16]
    int2* info;                              // per row: exponent, non-zero count
};

struct SplitArgs {
    Operand op[2];
    int64_t K;
    int nk, strips0;
};

constexpr int SPLIT_NT = 512, STRIP = 32;

// Exponent of each row's largest entry, then its digits. One CTA per strip
// of 32 rows: two passes over the strip (the second from L2), both along the
// operand's contiguous index; a thread writes 16 bytes (8 steps of K) of each
// plane, eight threads a whole 128-byte core matrix. Bound by HBM: 8 bytes
// read and 18 written per element.
__global__ void __launch_bounds__(SPLIT_NT) oz_split_kernel(SplitArgs a) {
    __shared__ unsigned smax[STRIP];
    __shared__ int scnt[STRIP];
    pdl_trigger();
    pdl_wait();
    const bool second = (int)blockIdx.x >= a.strips0;
    const Operand& o = a.op[second ? 1 : 0];
    const int64_t r0 = (int64_t)((int)blockIdx.x - (second ? a.strips0 : 0)) * STRIP;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    constexpr int NW = SPLIT_NT / 32;
    if (threadIdx.x < STRIP) {
        smax[threadIdx.x] = 0u;
        scnt[threadIdx.x] = 0;
    }
    __syncthreads();
    const int64_t ars = o.rs < 0 ? -o.rs : o.rs, als = o.ls < 0 ? -o.ls : o.ls;
    if (ars <= als) {                        // rows contiguous: a lane per row
        const int64_t r = r0 + lane;
        unsigned mx = 0;
        int cnt = 0;
        if (r < o.rows) {
            const double* src = o.X + r * o.rs;
#pragma unroll 8
            for (int64_t l = warp; l < a.K; l += NW) {
                const unsigned long long b = __double_as_longlong(src[l * o.ls]) &
                                             0x7fffffffffffffffull;
                mx = max(mx, (unsigned)(b >> 32));
                cnt += b != 0;
            }
            atomicMax(&smax[lane], mx);
            atomicAdd(&scnt[lane], cnt);
        }
    } else {                                 // K contiguous: lanes along K
        for (int q = warp; q < STRIP; q += NW) {
            const int64_t r = r0 + q;
            if (r >= o.rows) break;
            const double* src = o.X + r * o.rs;
            unsigned mx = 0;
            int cnt = 0;
#pragma unroll 8
            for (int64_t l = lane; l < a.K; l += 32) {
                const unsigned long long b = __double_as_longlong(src[l * o.ls]) &
                                             0x7fffffffffffffffull;
                mx = max(mx, (unsigned)(b >> 32));
                cnt += b != 0;
            }
            mx = __reduce_max_sync(0xffffffffu, mx);
            cnt = __reduce_add_sync(0xffffffffu, cnt);
            if (lane == 0) {
                smax[q] = mx;
                scnt[q] = cnt;
            }
        }
    }
    __syncthreads();
    const int64_t r = r0 + lane;
    if (r >= o.rows) return;
    const int emax = (int)(smax[lane] >> 20);
    if (warp == 0) {
        const int e = emax - 1021;           // |x| 2^-e < 1/2
        const bool ok = scnt[lane] == 0 || (e >= -kMaxExp && e <= kMaxExp);
        o.info[r] = make_int2(ok ? (scnt[lane] ? e : 0) : kBadExp, scnt[lane]);
    }
    const int64_t blk = r / o.br;
    const int rr = (int)(r - blk * o.br);
    const int64_t pb = plane_bytes(o.br);
    const double* src = o.X + r * o.rs;
    for (int kc = warp; kc < 2 * a.nk; kc += NW) {
        const int64_t l0 = (int64_t)kc * 8;
        unsigned lo[8], hi[8];               // lower seven digits, each + 128
        int top[8];
        unsigned mg[8];
        double x[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) x[u] = l0 + u < a.K ? __ldg(src + (l0 + u) * o.ls) : 0.0;
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const unsigned long long b = __double_as_longlong(x[u]);
            int ex = (int)(b >> 52) & 0x7ff;
            unsigned long long m = b & 0xfffffffffffffull;
            const int me = ex - emax + 125;  // magnitude as BF16, rounded down
            mg[u] = me > 0 && ex > 0 ? ((unsigned)me << 7) | (unsigned)(m >> 45) : 0u;
            if (ex > 0) m |= 1ull << 52;
            else ex = 1;
            const int sh = ex - emax + 10;   // x 2^(64 - e) = m 2^sh
            long long q;
            if (sh >= 0) q = (long long)(m << min(sh, 10));
            else if (sh < -54) q = 0;
            else q = (long long)((m + (1ull << (-sh - 1))) >> -sh);
            if (b >> 63) q = -q;
            const unsigned long long f =
                ((unsigned long long)q & 0xffffffffffffffull) + 0x80808080808080ull;
            top[u] = (int)(q >> 56) + (int)(f >> 56);
            lo[u] = (unsigned)f;
            hi[u] = (unsigned)(f >> 32);
        }
        const int ks = kc >> 1;
        const int64_t at = row_offset(rr) + (kc & 1) * 128;
        unsigned char* dst = o.digits + ((blk * a.nk + ks) * S) * pb + at;
#pragma unroll
        for (int s = 0; s < S; ++s) {
            unsigned w[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                float v[2];
#pragma unroll
                for (int t = 0; t < 2; ++t) {
                    const int z = 2 * u + t;
                    if (s == 0) {
                        v[t] = __int_as_float(0x4b400000 + top[z]) - 12582912.f;
                    } else {
                        const int byte = 7 - s;          // digit s + 1
                        const unsigned word = byte >= 4 ? hi[z] : lo[z];
                        v[t] = __uint_as_float(__byte_perm(word, 0x4b000000u,
                                                           0x7440 | (byte & 3))) -
                               8388736.f;
                    }
                }
                const __nv_bfloat162 p2 = __floats2bfloat162_rn(v[0], v[1]);
                w[u] = *reinterpret_cast<const unsigned*>(&p2);
            }
            *reinterpret_cast<uint4*>(dst + s * pb) = make_uint4(w[0], w[1], w[2], w[3]);
        }
        *reinterpret_cast<uint4*>(o.mags + (blk * a.nk + ks) * pb + at) =
            make_uint4(mg[0] | mg[1] << 16, mg[2] | mg[3] << 16, mg[4] | mg[5] << 16,
                       mg[6] | mg[7] << 16);
    }
}

struct Params {
    const unsigned char *pd, *pm, *qd, *qm;  // digit and magnitude images
    const int2 *pinfo, *qinfo;
    double* D;                               // D(r, c) = D[r * d_rs + c * d_cs]
    int64_t d_rs, d_cs, rows, cols;
    double beta, gamma;
    int nk, tm, tn;                          // K steps, tiles
    int* flags;                              // piece (r / 32, c / (BN / 2)): 1 = not done here
    int* err;
    long long wait_ns;
};

struct Smem {
    uint64_t full[STAGES], empty[STAGES], hi_full, hi_empty, lo_full, lo_empty, drain;
    uint32_t tmem_base;
    int abort;
};

using namespace tc;

__device__ bool wait_bounded(uint32_t bar, uint32_t parity, const Params& p, volatile int* abort,
                             bool honour_abort = true) {
    if (mbar_try(bar, parity)) return true;
    const uint64_t t0 = gtimer();
    const uint64_t limit = honour_abort ? (uint64_t)p.wait_ns
                                        : max((uint64_t)p.wait_ns, (uint64_t)1000000000ull);
    while (true) {
        if (mbar_try(bar, parity)) return true;
        if (honour_abort && *abort) return false;
        if (gtimer() - t0 > limit) {
            *abort = 1;
            atomicExch(p.err, kTimeout);
            return false;
        }
    }
}

__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes,
                                          uint32_t bar) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
        ::"r"(dst), "l"(src), "r"(bytes), "r"(bar)
        : "memory");
}

// Unswizzled K-major operand: core matrices of 8 rows x 16 bytes, the next
// one in K 128 bytes on, the next 8 rows 256 bytes on.
__device__ __forceinline__ uint64_t sdesc_plain(uint32_t saddr) {
    return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)(128 >> 4) << 16) |
           ((uint64_t)(256 >> 4) << 32) | ((uint64_t)1 << 46);
}

__device__ __forceinline__ void tmem_ld8(uint32_t taddr, float (&v)[8]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]),
                   "=f"(v[6]), "=f"(v[7])
                 : "r"(taddr));
}
__device__ __forceinline__ void tmem_wait_ld(float (&a)[8]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+f"(a[0]), "+f"(a[1]), "+f"(a[2]), "+f"(a[3]), "+f"(a[4]), "+f"(a[5]),
                   "+f"(a[6]), "+f"(a[7])
                 :
                 : "memory");
}
__device__ __forceinline__ void tmem_wait_ld(float (&a)[8], float (&b)[8], float (&c)[8],
                                             float (&d)[8]) {
    // the loaded registers pass through, so no use moves above the wait
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+f"(a[0]), "+f"(a[1]), "+f"(a[2]), "+f"(a[3]), "+f"(a[4]), "+f"(a[5]),
                   "+f"(a[6]), "+f"(a[7]), "+f"(b[0]), "+f"(b[1]), "+f"(b[2]), "+f"(b[3]),
                   "+f"(b[4]), "+f"(b[5]), "+f"(b[6]), "+f"(b[7])
                 :
                 : "memory");
    asm volatile(""
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3]), "+f"(c[4]), "+f"(c[5]),
                   "+f"(c[6]), "+f"(c[7]), "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3]),
                   "+f"(d[4]), "+f"(d[5]), "+f"(d[6]), "+f"(d[7])
                 :
                 : "memory");
}

template <int BN>
struct Cfg {
    static constexpr int A_PLANE = BM * KS * 2, B_PLANE = BN * KS * 2;
    static constexpr int A_BYTES = S * A_PLANE, B_BYTES = S * B_PLANE;
    static constexpr int STAGE_BYTES = A_BYTES + B_BYTES;
    static constexpr int TMEM_COLS = 8 * BN;             // one BN-column accumulator per level
    static constexpr int SMEM_BYTES = 1024 + STAGES * STAGE_BYTES + 256;
    static_assert(SMEM_BYTES <= 227 * 1024, "ring does not fit in shared memory");
    // kind::f16, FP32 accumulators, BF16 operands, both K-major, M = 128
    __host__ __device__ static constexpr uint32_t idesc(int n) {
        return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) |
               ((uint32_t)(BM >> 4) << 24);
    }
};

// Tile t: bands of 16 tile rows, column by column inside a band (operand
// panels shared in L2 by the tiles running together).
__device__ __forceinline__ void map_tile(const Params& p, int t, int& m, int& n) {
    constexpr int GM = 16;
    const int band = t / (GM * p.tn), first = band * GM, gm = min(GM, p.tm - first);
    const int idx = t - band * GM * p.tn;
    m = first + idx % gm;
    n = idx / gm;
}

// One CTA per SM, persistent over 128 x BN tiles. TMEM holds the eight level
// accumulators side by side, so the products of digit i with digits j .. j+3
// are ONE tcgen05.mma: the B planes of consecutive digits are consecutive rows
// in shared memory and their levels consecutive TMEM columns (N up to 256; 12
// instructions a K step instead of 36, and the A plane read 12 times instead
// of 36). Levels 2-5 ("hi") and 6-9 ("lo") are handed to the epilogue
// separately, and the steps of a chunk are issued in batches of two or three,
// all hi products before all lo ones: while the epilogue drains one group the
// tensor cores work on the other.
//
// Bound by the tensor pipe: 36 x 64 columns a step (1152 clocks at BN = 64)
// against 48 KB of operands through L2 and about 700 clocks of FP32 and integer
// work per drained step.
template <int BN>
__global__ void __launch_bounds__(NT, 1) oz_gemm_kernel(const __grid_constant__ Params p) {
    using C = Cfg<BN>;
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t ring = (raw + 1023u) & ~1023u;
    Smem* sm = reinterpret_cast<Smem*>(smem_raw + (ring - raw) + STAGES * C::STAGE_BYTES);
    volatile int* abort = &sm->abort;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(smem_u32(&sm->full[s]), 1);
            mbar_init(smem_u32(&sm->empty[s]), 1);
        }
        mbar_init(smem_u32(&sm->hi_full), 1);
        mbar_init(smem_u32(&sm->lo_full), 1);
        mbar_init(smem_u32(&sm->hi_empty), 8);
        mbar_init(smem_u32(&sm->lo_empty), 8);
        mbar_init(smem_u32(&sm->drain), 1);
        sm->abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         smem_u32(&sm->tmem_base)),
                     "r"(C::TMEM_COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = sm->tmem_base;
    pdl_trigger();
    pdl_wait();
    const int tiles = p.tm * p.tn;
    const int npm = (p.nk + S - 1) / S;      // magnitude stages: S steps each

    if (warp == 0 && lane == 0) {
        // ---------------- bulk-copy producer ----------------
        int stage = 0, issued = 0;
        uint32_t phase = 0;
        for (int t = blockIdx.x; t < tiles && !*abort; t += gridDim.x) {
            int m, n;
            map_tile(p, t, m, n);
            const unsigned char* pm = p.pm + (int64_t)m * p.nk * C::A_PLANE;
            const unsigned char* qm = p.qm + (int64_t)n * p.nk * C::B_PLANE;
            const unsigned char* pd = p.pd + (int64_t)m * p.nk * C::A_BYTES;
            const unsigned char* qd = p.qd + (int64_t)n * p.nk * C::B_BYTES;
            bool ok = true;
            for (int i = 0; i < npm + p.nk; ++i) {
                if (!wait_bounded(smem_u32(&sm->empty[stage]), phase ^ 1u, p, abort)) {
                    ok = false;
                    break;
                }
                const uint32_t fb = smem_u32(&sm->full[stage]);
                const uint32_t base = ring + stage * C::STAGE_BYTES;
                if (i < npm) {
                    const int ns = min(S, p.nk - i * S);
                    const uint32_t ab = (uint32_t)ns * C::A_PLANE, bb = (uint32_t)ns * C::B_PLANE;
                    mbar_expect_tx(fb, ab + bb);
                    bulk_load(base, pm + (int64_t)i * C::A_BYTES, ab, fb);
                    bulk_load(base + C::A_BYTES, qm + (int64_t)i * C::B_BYTES, bb, fb);
                } else {
                    const int ks = i - npm;
                    mbar_expect_tx(fb, C::STAGE_BYTES);
                    bulk_load(base, pd + (int64_t)ks * C::A_BYTES, C::A_BYTES, fb);
                    bulk_load(base + C::A_BYTES, qd + (int64_t)ks * C::B_BYTES, C::B_BYTES, fb);
                }
                ++issued;
                if (++stage == STAGES) { stage = 0; phase ^= 1u; }
            }
            if (!ok) break;
        }
        // Copies still in flight must land before the CTA exits.
        for (int i = 0; i < STAGES && i < issued; ++i) {
            if (--stage < 0) { stage = STAGES - 1; phase ^= 1u; }
            wait_bounded(smem_u32(&sm->full[stage]), phase, p, abort, false);
        }
    } else if (warp == 1 && lane == 0) {
        // ---------------- MMA issuer ----------------
        int stage = 0;
        uint32_t phase = 0, hi_phase = 0, lo_phase = 0;
        const auto wait_full = [&](int s, uint32_t ph) {
            if (!wait_bounded(smem_u32(&sm->full[s]), ph, p, abort)) return false;
            tc_fence_after();
            return true;
        };
        for (int t = blockIdx.x; t < tiles && !*abort; t += gridDim.x) {
            bool ok = wait_bounded(smem_u32(&sm->hi_empty), hi_phase ^ 1u, p, abort);
            if (!ok) break;
            tc_fence_after();
            // magnitudes: P in the columns of level 2
            for (int i = 0; i < npm && ok; ++i) {
                if (!(ok = wait_full(stage, phase))) break;
                const uint32_t a = ring + stage * C::STAGE_BYTES, b = a + C::A_BYTES;
                const int ns = min(S, p.nk - i * S);
                for (int s = 0; s < ns; ++s)
                    umma(tmem, sdesc_plain(a + s * C::A_PLANE), sdesc_plain(b + s * C::B_PLANE),
                         C::idesc(BN), (i | s) != 0 ? 1u : 0u);
                umma_commit(smem_u32(&sm->empty[stage]));
                if (++stage == STAGES) { stage = 0; phase ^= 1u; }
            }
            if (!ok) break;
            umma_commit(smem_u32(&sm->hi_full));
            hi_phase ^= 1u;
            for (int k0 = 0; k0 < p.nk && ok; k0 += CHUNK) {
                const int k1 = min(p.nk, k0 + CHUNK);
                for (int k = k0; k < k1 && ok;) {
                    const int left = k1 - k, nb = left == 4 ? 2 : min(3, left);
                    if (k == k0) {
                        if (!(ok = wait_bounded(smem_u32(&sm->hi_empty), hi_phase ^ 1u, p, abort)))
                            break;
                        tc_fence_after();
                    }
                    int s1 = stage;
                    uint32_t ph1 = phase;
                    for (int b = 0; b < nb && ok; ++b) {
                        if (!(ok = wait_full(s1, ph1))) break;
                        const uint32_t A = ring + s1 * C::STAGE_BYTES, B = A + C::A_BYTES;
                        const uint32_t on = k + b > k0 ? 1u : 0u;
#pragma unroll
                        for (int i = 1; i <= 4; ++i)     // levels i+1 .. 5: digits 1 .. 5-i of B
                            umma(tmem + (uint32_t)(BN * (i - 1)),
                                 sdesc_plain(A + (i - 1) * C::A_PLANE), sdesc_plain(B),
                                 C::idesc(BN * (5 - i)), i == 1 ? on : 1u);
                        if (++s1 == STAGES) { s1 = 0; ph1 ^= 1u; }
                    }
                    if (!ok) break;
                    if (k + nb == k1) umma_commit(smem_u32(&sm->hi_full));
                    if (k == k0) {
                        if (!(ok = wait_bounded(smem_u32(&sm->lo_empty), lo_phase ^ 1u, p, abort)))
                            break;
                        tc_fence_after();
                    }
                    for (int b = 0; b < nb; ++b) {
                        const uint32_t A = ring + stage * C::STAGE_BYTES, B = A + C::A_BYTES;
                        const uint32_t on = k + b > k0 ? 1u : 0u;
#pragma unroll
                        for (int i = 1; i <= 8; ++i) {   // levels max(6, i+1) .. 9
                            const int j0 = i < 6 ? 6 - i : 1, j1 = 9 - i;
                            umma(tmem + (uint32_t)(BN * (i + j0 - 2)),
                                 sdesc_plain(A + (i - 1) * C::A_PLANE),
                                 sdesc_plain(B + (j0 - 1) * C::B_PLANE),
                                 C::idesc(BN * (j1 - j0 + 1)), i == 1 ? on : 1u);
                        }
                        umma_commit(smem_u32(&sm->empty[stage]));
                        if (++stage == STAGES) { stage = 0; phase ^= 1u; }
                    }
                    k += nb;
                }
                if (!ok) break;
                umma_commit(smem_u32(&sm->lo_full));
                hi_phase ^= 1u;
                lo_phase ^= 1u;
            }
            if (!ok) break;
        }
        // All MMAs issued by this CTA complete before TMEM is released.
        umma_commit(smem_u32(&sm->drain));
        wait_bounded(smem_u32(&sm->drain), 0, p, abort, false);
    } else if (warp >= 2) {
        // ---------------- epilogue ----------------
        // warp w: TMEM lanes 32 (w % 4) .., columns [half * HC, half * HC + HC)
        constexpr int HC = BN / 2;
        const int q = warp & 3, half = (warp - 2) >> 2;
        const uint32_t tq = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(half * HC);
        uint32_t hi_phase = 0, lo_phase = 0;
        const auto warp_wait = [&](uint64_t* bar, uint32_t ph) {
            int w = 1;
            if (lane == 0) w = wait_bounded(smem_u32(bar), ph, p, abort);
            w = __shfl_sync(0xffffffffu, w, 0);
            tc_fence_after();
            return w != 0;
        };
        const auto release = [&](uint64_t* bar) {
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(bar));
        };
        constexpr float kMagic = 12582912.f;             // 1.5 2^23
        for (int t = blockIdx.x; t < tiles; t += gridDim.x) {
            int m, n;
            map_tile(p, t, m, n);
            const int64_t row = (int64_t)m * BM + q * 32 + lane;
            const int64_t col0 = (int64_t)n * BN + half * HC;
            const bool row_ok = row < p.rows;
            const int2 ri = row_ok ? p.pinfo[row] : make_int2(0, 0);
            int bad = ri.x == kBadExp;
            if (!warp_wait(&sm->hi_full, hi_phase)) break;
            hi_phase ^= 1u;
#pragma unroll 1
            for (int c = 0; c < HC; c += 8) {
                float v[8];
                tmem_ld8(tq + c, v);
                tmem_wait_ld(v);
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    if (col0 + c + u < p.cols && row_ok) {
                        const int2 ci = __ldg(p.qinfo + col0 + c + u);
                        const int cnt = min(ri.y, ci.y);
                        bad |= ci.x == kBadExp ||
                               (cnt > 0 && !(v[u] >= (float)cnt * 0x1p-12f));
                    }
                }
            }
            release(&sm->hi_empty);
            bad = __any_sync(0xffffffffu, bad);
            // running sums: T in units of level 6, R in units of level 8. The
            // magic constants that turn levels 2 and 3 into integers come off
            // here, once for all chunks.
            const long long nch = (p.nk + CHUNK - 1) / CHUNK;
            const long long t0 = (long long)(0ull - (unsigned long long)nch *
                                                        ((0x4b400000ull << 24) + (0x4b400000ull << 32)));
            long long T[HC];
            float R[HC];
#pragma unroll
            for (int c = 0; c < HC; ++c) {
                T[c] = t0;
                R[c] = 0.f;
            }
            bool ok = true;
            for (int k0 = 0; k0 < p.nk; k0 += CHUNK) {
                if (!(ok = warp_wait(&sm->hi_full, hi_phase))) break;
                hi_phase ^= 1u;
#pragma unroll
                for (int c = 0; c < HC; c += 8) {
                    float l2[8], l3[8], l4[8], l5[8];
                    tmem_ld8(tq + c, l2);
                    tmem_ld8(tq + BN + c, l3);
                    tmem_ld8(tq + 2 * BN + c, l4);
                    tmem_ld8(tq + 3 * BN + c, l5);
                    tmem_wait_ld(l2, l3, l4, l5);
#pragma unroll
                    for (int u = 0; u < 8; ++u) {
                        long long x = T[c + u];
                        x += (long long)__float2int_rn(l5[u]) << 8;
                        x += (long long)__float2int_rn(l4[u]) << 16;
                        // |level 3| <= 2^22, |level 2| <= 2^21
                        x += (long long)((unsigned long long)__float_as_uint(l3[u] + kMagic) << 24);
                        x += (long long)((unsigned long long)__float_as_uint(l2[u] + kMagic) << 32);
                        T[c + u] = x;
                    }
                }
                release(&sm->hi_empty);
                if (!(ok = warp_wait(&sm->lo_full, lo_phase))) break;
                lo_phase ^= 1u;
#pragma unroll
                for (int c = 0; c < HC; c += 8) {
                    float l6[8], l7[8], l8[8], l9[8];
                    tmem_ld8(tq + 4 * BN + c, l6);
                    tmem_ld8(tq + 5 * BN + c, l7);
                    tmem_ld8(tq + 6 * BN + c, l8);
                    tmem_ld8(tq + 7 * BN + c, l9);
                    tmem_wait_ld(l6, l7, l8, l9);
#pragma unroll
                    for (int u = 0; u < 8; ++u) {
                        // carries of 256 from level 8 into 7 and from 7 into 6
                        const float g8 = fmaf(l9[u], 0x1p-8f, l8[u]);
                        const float t8 = fmaf(g8, 0x1p-8f, kMagic) - kMagic;
                        const float g7 = l7[u] + t8;
                        const float t7 = fmaf(g7, 0x1p-8f, kMagic) - kMagic;
                        R[c + u] += fmaf(t8, -256.f, g8);
                        R[c + u] = fmaf(fmaf(t7, -256.f, g7), 256.f, R[c + u]);
                        T[c + u] += __float2int_rn(l6[u] + t7);
                    }
                }
                release(&sm->lo_empty);
            }
            if (!ok) break;
            const int64_t pieces = (int64_t)p.tn * 2;
            if (lane == 0 && row < p.rows && col0 < p.cols)
                p.flags[((int64_t)m * 4 + q) * pieces + n * 2 + half] = bad;
            if (bad || !row_ok) continue;
            // T 2^-48 + R 2^-64 as one double (units 2^-64), rounded once:
            // 2^100 + (T >> 32) 2^48 less its offset, plus the low 32 bits and R
            // in the mantissa of 2^52
            const double g = p.gamma * __hiloint2double((1023 + ri.x - 64) << 20, 0);
            double* dst = p.D + row * p.d_rs + col0 * p.d_cs;
#pragma unroll
            for (int c = 0; c < HC; ++c) {
                if (col0 + c < p.cols) {
                    const int th = (int)(T[c] >> 32);
                    const unsigned tl = (unsigned)T[c];
                    const double da = __hiloint2double(0x46300000, th ^ (int)0x80000000);
                    const unsigned long long mb = 0x4338000000000000ull +
                                                  ((unsigned long long)tl << 16) +
                                                  (unsigned long long)(long long)__float2int_rn(R[c]);
                    const double v = (da - (0x1p100 + 0x1p79 + 0x1p52 + 0x1p51)) +
                                     __longlong_as_double((long long)mb);
                    const int ce = __ldg(p.qinfo + col0 + c).x;
                    const double vs =
                        v == 0.0 ? 0.0 : __hiloint2double(__double2hiint(v) + (ce << 20),
                                                         __double2loint(v));
                    double* d = dst + c * p.d_cs;
                    *d = fma(g, vs, p.beta == 1.0 ? *d : p.beta * *d);
                }
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 1) {
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                     "r"(C::TMEM_COLS)
                     : "memory");
    }
}

inline int64_t up(int64_t x, int64_t q) { return (x + q - 1) / q * q; }

// Byte layout of one update's scratch.
struct Layout {
    size_t pd, pm, qd, qm, pi, qi, flags, total;
};
static Layout layout(int64_t rows, int64_t cols, int64_t K) {
    const int64_t nk = (K + KS - 1) / KS, pr = up(rows, BM), qr = up(cols, 64);
    Layout w;
    size_t at = 0;
    const auto take = [&](int64_t bytes) {
        const size_t o = at;
        at += (size_t)up(bytes, 256);
        return o;
    };
    w.pd = take(pr * nk * KS * 2 * S);
    w.pm = take(pr * nk * KS * 2);
    w.qd = take(qr * nk * KS * 2 * S);
    w.qm = take(qr * nk * KS * 2);
    w.pi = take(pr * (int64_t)sizeof(int2));
    w.qi = take(qr * (int64_t)sizeof(int2));
    w.flags = take(pr / 32 * (qr / 8) * (int64_t)sizeof(int));
    w.total = at;
    return w;
}

}  // namespace oz

cudaError_t oz_configure() {
    cudaError_t e;
    if ((e = cudaFuncSetAttribute(oz::oz_gemm_kernel<64>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  oz::Cfg<64>::SMEM_BYTES)) != cudaSuccess)
        return e;
    if ((e = cudaFuncSetAttribute(oz::oz_gemm_kernel<32>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  oz::Cfg<32>::SMEM_BYTES)) != cudaSuccess)
        return e;
    return cudaFuncSetAttribute(oz::oz_gemm_kernel<16>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                oz::Cfg<16>::SMEM_BYTES);
}

size_t oz_update_bytes(int64_t mlen, int64_t nrhs, int64_t klen) {
    // either orientation (the tile's 128 rows lie along C's contiguous index)
    return std::max(oz::layout(mlen, nrhs, klen).total, oz::layout(nrhs, mlen, klen).total);
}

cudaError_t launch_oz_update(const Canon<double>& p, const TcGemm& g, double beta, double gamma,
                             void* ws, int* err, long long wait_ns, int num_sms, cudaStream_t s) {
    using namespace oz;
    // tile rows (TMEM lanes) along C's contiguous index: the epilogue's lanes
    // then read and write whole lines of C
    const bool swap = (p.c_cs == 1 || p.c_cs == -1) && p.c_rs != 1 && p.c_rs != -1;
    const int64_t rows = swap ? p.nrhs : g.mlen, cols = swap ? g.mlen : p.nrhs;
    const int64_t tm = (rows + BM - 1) / BM;
    // the widest tile that still gives every SM one
    const int bn = tm * ((cols + 63) / 64) >= num_sms ? 64 : tm * ((cols + 31) / 32) >= num_sms ? 32 : 16;
    const Layout w = layout(rows, cols, g.klen);
    unsigned char* base = static_cast<unsigned char*>(ws);
    SplitArgs a;
    Operand M, Y;
    M.X = p.A + g.rc * p.a_rs + g.rk * p.a_cs;
    M.rs = p.a_rs;
    M.ls = p.a_cs;
    M.rows = g.mlen;
    Y.X = p.C + g.rk * p.c_rs;
    Y.rs = p.c_cs;
    Y.ls = p.c_rs;
    Y.rows = p.nrhs;
    a.op[0] = swap ? Y : M;
    a.op[1] = swap ? M : Y;
    a.op[0].br = BM;
    a.op[0].digits = base + w.pd;
    a.op[0].mags = base + w.pm;
    a.op[0].info = reinterpret_cast<int2*>(base + w.pi);
    a.op[1].br = bn;
    a.op[1].digits = base + w.qd;
    a.op[1].mags = base + w.qm;
    a.op[1].info = reinterpret_cast<int2*>(base + w.qi);
    a.K = g.klen;
    a.nk = (int)((g.klen + KS - 1) / KS);
    a.strips0 = (int)((rows + STRIP - 1) / STRIP);
    const int64_t strips = a.strips0 + (cols + STRIP - 1) / STRIP;
    cudaError_t e = launch_kernel(oz_split_kernel, dim3((unsigned)strips), dim3(SPLIT_NT), 0, s, a);
    if (e != cudaSuccess) return e;
    Params q;
    q.pd = a.op[0].digits;
    q.pm = a.op[0].mags;
    q.qd = a.op[1].digits;
    q.qm = a.op[1].mags;
    q.pinfo = a.op[0].info;
    q.qinfo = a.op[1].info;
    q.D = p.C + g.rc * p.c_rs;
    q.d_rs = swap ? p.c_cs : p.c_rs;
    q.d_cs = swap ? p.c_rs : p.c_cs;
    q.rows = rows;
    q.cols = cols;
    q.beta = beta;
    q.gamma = gamma;
    q.nk = a.nk;
    q.tm = (int)tm;
    q.tn = (int)((cols + bn - 1) / bn);
    q.flags = reinterpret_cast<int*>(base + w.flags);
    q.err = err;
    q.wait_ns = wait_ns;
    const int64_t tiles = (int64_t)q.tm * q.tn;
    if (tiles > (int64_t)1 << 30) return cudaErrorInvalidValue;
    const dim3 grid((unsigned)std::min<int64_t>(tiles, num_sms));
    e = bn == 64   ? launch_kernel(oz_gemm_kernel<64>, grid, dim3(NT), Cfg<64>::SMEM_BYTES, s, q)
        : bn == 32 ? launch_kernel(oz_gemm_kernel<32>, grid, dim3(NT), Cfg<32>::SMEM_BYTES, s, q)
                   : launch_kernel(oz_gemm_kernel<16>, grid, dim3(NT), Cfg<16>::SMEM_BYTES, s, q);
    if (e != cudaSuccess) return e;
    OzPieces pc;
    pc.flags = q.flags;
    pc.per_row = (int64_t)q.tn * 2;
    pc.cols = bn / 2;
    pc.swap = swap;
    return launch_gemm_simt_pieces(p, g.rc, g.mlen, g.rk, g.klen, beta, gamma, pc, s, num_sms);
}

}  // namespace trx
