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
// and, from the same pieces, the whole triangular product (TRMM) and the
// residual of refinement, B - M X, as one launch each.
//
// Arithmetic. Each row of either operand (over a segment of at most 4096 of K)
// is scaled by a power of two to below 1/2 in magnitude and rounded to a 64-bit
// fixed-point number, whose eight balanced base-256 digits d_1 .. d_8 (weights
// 2^-8 .. 2^-64, each in [-128, 128]) are exact in BF16. The products of digits i
// and j with i + j <= 9 are summed on the tensor cores, one FP32 accumulator per
// weight 2^-8(i+j) ("level" 2 .. 9). Over K chunks of 192 the levels 2-6 are sums
// of at most 5 * 192 products of two digits, below 2^24 and so exact integers;
// levels 7-9 (weight 2^-56 and less) can pass 2^24, and be rounded by a few units,
// only where nearly all digits are near 128 (P is then above K' / 40). Chunks are
// added up exactly in 64-bit integers (levels 2-6) and in FP32 values of two
// digits (levels 7-8, level 9 rounded to 2^-64). Left out: the digit products of
// i + j >= 10, below 0.88 2^-63 a term; the rounding of the operands adds 0.25 2^-63 and
// that of level 9 as much a chunk. In units of the scaled operands a segment's
// error is below K' 2^-62, K' the smaller count of non-zeros of the two rows.
//
// When it applies. That error is relative to the rows' largest entries, not
// to sum |m||c| as an FMA chain's is. So the kernel also forms P = |M||C| (one
// BF16 product of the rounded-down magnitudes, 3 % more work) and keeps the
// sum of a 32-row x BN/2-column piece only where P >= K' 2^-12 for every
// element, i.e. where its error is below 8 u sum |m||c| (u = 2^-53; the bound
// of a K-term FMA chain is K u sum |m||c|). The sums of pieces that fail, or that
// hold an Inf, a NaN or a row outside 2^+-300, are not added but flagged, and
// the DFMA kernel (gemm_simt.cu), launched after this one over the flagged
// pieces only, adds them. The residual takes pieces with P >= K' 2^-16 (error
// below 2^-46 sum |m||x|, the float-float residual's).
//
// Measured, 2048 x 4096 with K 2048 (operand split, product and the empty DFMA
// pass together): 897 us, 38 TFLOP/s, against 28567 us by DFMA; 4096^3 44
// TFLOP/s (1.6 PFLOP/s of BF16 products). Relative error against quad precision
// 5.6e-17 (DFMA 7.7e-16).
#include <stdint.h>

#include <algorithm>

#include "common.cuh"
#include "tc_ptx.cuh"

namespace trx {
namespace oz {

constexpr int S = 8;                         // digits per operand
constexpr int BM = 128;                      // rows of a tile (TMEM lanes)
constexpr int KS = 16;                       // K of one step (one tcgen05.mma)
constexpr int CHUNK = 12;                    // steps per exact sum (192 terms)
constexpr int STAGES = 4;                    // ring depth, one step per stage
// One warpgroup of producer and MMA issuer, two of epilogue warps. The kernel
// launches with 168 registers a thread; the first warpgroup keeps 56 and the
// others take 224 (128 * 56 + 256 * 224 = 384 * 168), which holds a thread's
// running sums and 16 columns of four levels without spills.
constexpr int NT = 384, REGS_ISSUE = 56, REGS_EPILOGUE = 224;
static_assert(128 * REGS_ISSUE + 256 * REGS_EPILOGUE <= NT * 168, "register split");
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

// Segments of K with a scale of their own: a row whose entries grow or decay
// over K keeps its digits where it is small.
constexpr int SEG = 4096, SEG_STEPS = SEG / KS;
__host__ __device__ constexpr int nseg(int64_t K) { return (int)((K + SEG - 1) / SEG); }

struct Operand {                             // element (r, l) = X[r * rs + l * ls]
    const void* X;
    int64_t rs, ls, rows;
    int br;                                  // rows per block
    int tri;                                 // 1: only l < r; blocks end with their last row
    unsigned char* digits;                   // [block][step][digit][br x 16]
    unsigned char* mags;                     // [block][step][br x 16]
    int2* info;                              // [segment][row]: exponent, non-zero count
    double* copy;                            // optional copy, (r, l) at r * K + l
};
// Steps of K before block b of an operand, and in it.
__host__ __device__ inline int64_t steps_before(int tri, int br, int64_t b, int64_t nk) {
    return tri ? br / KS * (b * (b + 1) / 2) : b * nk;
}
__host__ __device__ inline int steps_in(int tri, int br, int64_t b, int64_t nk) {
    const int64_t t = (b + 1) * (br / KS);
    return (int)(tri && t < nk ? t : nk);
}

struct SplitArgs {
    Operand op[2];
    int64_t K;
    int nk, strips0;
};

constexpr int SPLIT_NT = 256, STRIP = 16;

// Exponent of each row's largest entry, then its digits. One CTA per strip
// of 16 rows (inside one block) and segment: two passes over it (the second from
// L1 and L2), both along the operand's contiguous index; a thread writes 16 bytes
// (8 of K) of each plane, a warp 16 rows x one K step: 512 consecutive bytes.
// Bound by HBM at large sizes (8 bytes read, 18 written per element) and by the
// load latency of its few rounds at small ones; strips of 16 rows and 256 threads
// in place of 32 and 512 keep twice the CTAs in flight: 19 -> 11
// us for 512 x 200 with K 512, 112 -> 93 for 2048 x 4096 with K 2048.
template <typename TX>
__device__ void split_strip(const Operand& o, int64_t K, int nk, int64_t r0) {
    __shared__ unsigned smax[STRIP];
    __shared__ int scnt[STRIP];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int rl = lane & (STRIP - 1), kl = lane / STRIP;
    constexpr int NW = SPLIT_NT / 32, KL = 32 / STRIP;
    const TX* X = static_cast<const TX*>(o.X);
    const int seg = blockIdx.y;
    const int64_t k0 = (int64_t)seg * SEG, k1 = min(K, k0 + SEG);
    if (o.tri && k0 >= (r0 / o.br + 1) * o.br) return;
    if (threadIdx.x < STRIP) {
        smax[threadIdx.x] = 0u;
        scnt[threadIdx.x] = 0;
    }
    __syncthreads();
    const int64_t r = r0 + rl;
    const int64_t ars = o.rs < 0 ? -o.rs : o.rs, als = o.ls < 0 ? -o.ls : o.ls;
    if (ars <= als) {                        // rows contiguous: a lane per row
        unsigned mx = 0;
        int cnt = 0;
        if (r < o.rows) {
            const TX* src = X + r * o.rs;
            const int64_t end = o.tri ? min(k1, r) : k1;
#pragma unroll 8
            for (int64_t l = k0 + warp * KL + kl; l < end; l += NW * KL) {
                const unsigned long long b = __double_as_longlong((double)src[l * o.ls]) &
                                             0x7fffffffffffffffull;
                mx = max(mx, (unsigned)(b >> 32));
                cnt += b != 0;
            }
            atomicMax(&smax[rl], mx);
            atomicAdd(&scnt[rl], cnt);
        }
    } else {                                 // K contiguous: lanes along K
        for (int q = warp; q < STRIP; q += NW) {
            if (r0 + q >= o.rows) break;
            const TX* src = X + (r0 + q) * o.rs;
            const int64_t end = o.tri ? min(k1, r0 + q) : k1;
            unsigned mx = 0;
            int cnt = 0;
#pragma unroll 16
            for (int64_t l = k0 + lane; l < end; l += 32) {
                const unsigned long long b = __double_as_longlong((double)src[l * o.ls]) &
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
    if (r >= o.rows) return;
    const int emax = (int)(smax[rl] >> 20);
    if (warp == 0 && kl == 0 && blockIdx.z == 0) {
        const int e = emax - 1021;           // |x| 2^-e < 1/2
        const bool ok = scnt[rl] == 0 || (e >= -kMaxExp && e <= kMaxExp);
        o.info[seg * o.rows + r] = make_int2(ok ? (scnt[rl] ? e : 0) : kBadExp, scnt[rl]);
    }
    const int64_t blk = r / o.br;
    const int rr = (int)(r - blk * o.br);
    const int64_t pb = plane_bytes(o.br), sb = steps_before(o.tri, o.br, blk, nk);
    const int kc1 = 2 * min(steps_in(o.tri, o.br, blk, nk), (seg + 1) * SEG_STEPS);
    const int64_t end = o.tri ? r : K;       // entries from here on are zero
    const TX* src = X + r * o.rs;
    // 16-byte loads of FP64 data along K where every row starts on 16 bytes
    const bool pairs = sizeof(TX) == 8 && o.ls == 1 && (o.rs & 1) == 0 &&
                       (reinterpret_cast<uintptr_t>(X) & 15) == 0;
    for (int kc = 2 * seg * SEG_STEPS + ((int)blockIdx.z * NW + warp) * KL + kl; kc < kc1;
         kc += (int)gridDim.z * NW * KL) {
        const int64_t l0 = (int64_t)kc * 8;
        unsigned lo[8], hi[8];               // lower seven digits, each + 128
        int top[8];
        unsigned mg[8];
        double x[8];
        if (pairs && l0 + 8 <= end) {
#pragma unroll
            for (int u = 0; u < 8; u += 2) {
                const double2 v = __ldg(reinterpret_cast<const double2*>(src + l0 + u));
                x[u] = v.x;
                x[u + 1] = v.y;
            }
        } else {
#pragma unroll
            for (int u = 0; u < 8; ++u)
                x[u] = l0 + u < end ? (double)__ldg(src + (l0 + u) * o.ls) : 0.0;
        }
        if (o.copy) {
#pragma unroll
            for (int u = 0; u < 8; ++u)
                if (l0 + u < end) o.copy[r * K + l0 + u] = x[u];
        }
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
        const int64_t ks = sb + (kc >> 1);
        const int64_t at = row_offset(rr) + (kc & 1) * 128;
        unsigned char* dst = o.digits + ks * S * pb + at;
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
        *reinterpret_cast<uint4*>(o.mags + ks * pb + at) =
            make_uint4(mg[0] | mg[1] << 16, mg[2] | mg[3] << 16, mg[4] | mg[5] << 16,
                       mg[6] | mg[7] << 16);
    }
}

// Operand 0 of type T0 (strips [0, strips0)), operand 1 double.
template <typename T0>
__global__ void __launch_bounds__(SPLIT_NT, 2) oz_split_kernel(SplitArgs a) {
    pdl_trigger();
    pdl_wait();
    const int s = blockIdx.x;
    if (s < a.strips0) split_strip<T0>(a.op[0], a.K, a.nk, (int64_t)s * STRIP);
    else split_strip<double>(a.op[1], a.K, a.nk, (int64_t)(s - a.strips0) * STRIP);
}

// D(r, c) := c0 E(r, c) + dg d(i) F(r, c) + gamma sum, i the triangle's row (r, or
// c when tri == 2); E or F may be null (no such term), or D itself.
struct Params {
    const unsigned char *pd, *pm, *qd, *qm;  // digit and magnitude images
    const int2 *pinfo, *qinfo;
    double* D;                               // D(r, c) = D[r * d_rs + c * d_cs]
    int64_t d_rs, d_cs, rows, cols;
    const double* E;
    int64_t e_rs, e_cs;
    double c0;
    const double* F;
    int64_t f_rs, f_cs;
    double dg;
    const void* diag;                        // d(i) = diag[i * d_step], 1 when null
    int64_t d_step;
    int diag_f32;
    double gamma;
    float least;                             // a piece needs P >= least * K'
    int tri;                                 // triangular operand: 0 none, 1 P, 2 Q
    int nk, tm, tn, band;                    // K steps, tiles, raster band
    int* flags;                              // [segment] piece (r / 32, c / (BN / 2)): 1 = sum
    int64_t seg_flags;                       // not added here; flags per segment
    int* err;
    long long wait_ns;
};

__device__ __forceinline__ double diagonal(const Params& p, int64_t i) {
    if (!p.diag) return 1.0;
    return p.diag_f32 ? (double)__ldg(static_cast<const float*>(p.diag) + i * p.d_step)
                      : __ldg(static_cast<const double*>(p.diag) + i * p.d_step);
}

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

// W columns of 32 lanes (W = 8 or 16), not waited for.
template <int W>
__device__ __forceinline__ void tmem_ld(uint32_t taddr, float (&v)[W]) {
    if constexpr (W == 16) {
        asm volatile(
            "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
            "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
            : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]),
              "=f"(v[7]), "=f"(v[8]), "=f"(v[9]), "=f"(v[10]), "=f"(v[11]), "=f"(v[12]),
              "=f"(v[13]), "=f"(v[14]), "=f"(v[15])
            : "r"(taddr));
    } else {
        static_assert(W == 8, "8 or 16 columns");
        asm volatile(
            "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
            : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]),
              "=f"(v[7])
            : "r"(taddr));
    }
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

// Tile t: bands of p.band tile rows (tri == 2: columns), across inside a band, so
// the tiles running together share operand panels in L2; a triangle's longest
// rows first.
__device__ __forceinline__ void map_tile(const Params& p, int t, int& m, int& n) {
    const int to = p.tri == 2 ? p.tn : p.tm, ti = p.tri == 2 ? p.tm : p.tn;
    const int band = t / (p.band * ti), first = band * p.band, g = min(p.band, to - first);
    const int idx = t - band * p.band * ti;
    const int o = first + idx % g, i = idx / g;
    m = p.tri == 2 ? i : p.tri == 1 ? p.tm - 1 - o : o;
    n = p.tri == 2 ? p.tn - 1 - o : i;
}
// Rounds run alternately forwards and backwards over the CTAs (rows of
// unequal length even out).
__device__ __forceinline__ int round_tile(int r) {
    const int c = (r & 1) ? (int)(gridDim.x - 1 - blockIdx.x) : (int)blockIdx.x;
    return r * (int)gridDim.x + c;
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
// Bound by the tensor pipe at BN = 64: 36 x 64 columns a step (1184 clocks) against 48
// KB of operands through L2; 70 % active at 4096^3, and 40 % at BN = 32, whose MMAs are at
// their least time. One lane, elect.sync's, waits, issues and
// commits: FP64 TRSM 4096 x 4096 5205 us, TRMM 2500 x 1500 455; with lane 0 in its place
// 5353 and 485.
template <int BN>
__global__ void __launch_bounds__(NT, 1) oz_gemm_kernel(const __grid_constant__ Params p) {
    using C = Cfg<BN>;
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t ring = (raw + 1023u) & ~1023u;
    Smem* sm = reinterpret_cast<Smem*>(smem_raw + (ring - raw) + STAGES * C::STAGE_BYTES);
    volatile int* abort = &sm->abort;
    const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
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
    const uint32_t tmem = __shfl_sync(0xffffffffu, sm->tmem_base, 0);
    pdl_trigger();
    pdl_wait();
    const int tiles = p.tm * p.tn;
    // K steps of a tile (a triangle's row ends with its last row)
    const auto tile_steps = [&](int m, int n) {
        return p.tri == 1   ? steps_in(1, BM, m, p.nk)
               : p.tri == 2 ? steps_in(1, BN, n, p.nk)
                            : p.nk;
    };

    if (warp < 4) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(REGS_ISSUE));
        if (warp == 0 && lane == 0) {
            // ---------------- bulk-copy producer ----------------
            int stage = 0, issued = 0;
            uint32_t phase = 0;
            bool ok = true;
            for (int r = 0, t; ok && (t = round_tile(r)) < tiles && !*abort; ++r) {
                int m, n;
                map_tile(p, t, m, n);
                const int nk = tile_steps(m, n);
                const int64_t ps = steps_before(p.tri == 1, BM, m, p.nk);
                const int64_t qs = steps_before(p.tri == 2, BN, n, p.nk);
                for (int s0 = 0; s0 < nk && ok; s0 += SEG_STEPS) {
                    const int sn = min(SEG_STEPS, nk - s0), npm = (sn + S - 1) / S;
                    const unsigned char* pm = p.pm + (ps + s0) * C::A_PLANE;
                    const unsigned char* qm = p.qm + (qs + s0) * C::B_PLANE;
                    const unsigned char* pd = p.pd + (ps + s0) * C::A_BYTES;
                    const unsigned char* qd = p.qd + (qs + s0) * C::B_BYTES;
                    for (int i = 0; i < npm + sn; ++i) {
                        if (!wait_bounded(smem_u32(&sm->empty[stage]), phase ^ 1u, p, abort)) {
                            ok = false;
                            break;
                        }
                        const uint32_t fb = smem_u32(&sm->full[stage]);
                        const uint32_t base = ring + stage * C::STAGE_BYTES;
                        if (i < npm) {           // magnitudes: S steps a stage
                            const int ns = min(S, sn - i * S);
                            const uint32_t ab = (uint32_t)ns * C::A_PLANE;
                            const uint32_t bb = (uint32_t)ns * C::B_PLANE;
                            mbar_expect_tx(fb, ab + bb);
                            bulk_load(base, pm + (int64_t)i * C::A_BYTES, ab, fb);
                            bulk_load(base + C::A_BYTES, qm + (int64_t)i * C::B_BYTES, bb, fb);
                        } else {
                            const int ks = i - npm;
                            mbar_expect_tx(fb, C::STAGE_BYTES);
                            bulk_load(base, pd + (int64_t)ks * C::A_BYTES, C::A_BYTES, fb);
                            bulk_load(base + C::A_BYTES, qd + (int64_t)ks * C::B_BYTES, C::B_BYTES,
                                      fb);
                        }
                        ++issued;
                        if (++stage == STAGES) { stage = 0; phase ^= 1u; }
                    }
                }
            }
            // Copies still in flight must land before the CTA exits.
            for (int i = 0; i < STAGES && i < issued; ++i) {
                if (--stage < 0) { stage = STAGES - 1; phase ^= 1u; }
                wait_bounded(smem_u32(&sm->full[stage]), phase, p, abort, false);
            }
        } else if (warp == 1 && elect_lane()) {
            // ---------------- MMA issuer ----------------
            int stage = 0;
            uint32_t phase = 0, hi_phase = 0, lo_phase = 0;
            const uint64_t a_ring = sdesc_plain(ring), b_ring = sdesc_plain(ring + C::A_BYTES);
            constexpr uint32_t ST = C::STAGE_BYTES >> 4, AP = C::A_PLANE >> 4, BP = C::B_PLANE >> 4;
            const auto wait = [&](uint64_t* bar, uint32_t ph, bool honour_abort = true) {
                if (!wait_bounded(smem_u32(bar), ph, p, abort, honour_abort)) return false;
                tc_fence_after();
                return true;
            };
            const auto segment = [&](int nk) {
                if (!wait(&sm->hi_empty, hi_phase ^ 1u)) return false;
                const int npm = (nk + S - 1) / S;
                // magnitudes: P in the columns of level 2
                for (int i = 0; i < npm; ++i) {
                    if (!wait(&sm->full[stage], phase)) return false;
                    const uint64_t a = a_ring + stage * ST, b = b_ring + stage * ST;
                    const int ns = min(S, nk - i * S);
                    for (int s = 0; s < ns; ++s)
                        umma(tmem, a + s * AP, b + s * BP, C::idesc(BN), (i | s) != 0 ? 1u : 0u);
                    umma_commit(smem_u32(&sm->empty[stage]));
                    if (++stage == STAGES) { stage = 0; phase ^= 1u; }
                }
                umma_commit(smem_u32(&sm->hi_full));
                hi_phase ^= 1u;
                for (int k0 = 0; k0 < nk; k0 += CHUNK) {
                    const int k1 = min(nk, k0 + CHUNK);
                    for (int k = k0; k < k1;) {
                        const int left = k1 - k, nb = left == 4 ? 2 : min(3, left);
                        if (k == k0 && !wait(&sm->hi_empty, hi_phase ^ 1u)) return false;
                        int s1 = stage;
                        uint32_t ph1 = phase;
                        for (int b = 0; b < nb; ++b) {
                            if (!wait(&sm->full[s1], ph1)) return false;
                            const uint64_t A = a_ring + s1 * ST, B = b_ring + s1 * ST;
                            const uint32_t on = k + b > k0 ? 1u : 0u;
#pragma unroll
                            for (int i = 1; i <= 4; ++i)     // levels i+1 .. 5: B digits 1 .. 5-i
                                umma(tmem + (uint32_t)(BN * (i - 1)), A + (i - 1) * AP, B,
                                     C::idesc(BN * (5 - i)), i == 1 ? on : 1u);
                            if (++s1 == STAGES) { s1 = 0; ph1 ^= 1u; }
                        }
                        if (k + nb == k1) umma_commit(smem_u32(&sm->hi_full));
                        if (k == k0 && !wait(&sm->lo_empty, lo_phase ^ 1u)) return false;
                        for (int b = 0; b < nb; ++b) {
                            const uint64_t A = a_ring + stage * ST, B = b_ring + stage * ST;
                            const uint32_t on = k + b > k0 ? 1u : 0u;
#pragma unroll
                            for (int i = 1; i <= 8; ++i) {   // levels max(6, i+1) .. 9
                                const int j0 = i < 6 ? 6 - i : 1, j1 = 9 - i;
                                umma(tmem + (uint32_t)(BN * (i + j0 - 2)), A + (i - 1) * AP,
                                     B + (j0 - 1) * BP, C::idesc(BN * (j1 - j0 + 1)),
                                     i == 1 ? on : 1u);
                            }
                            umma_commit(smem_u32(&sm->empty[stage]));
                            if (++stage == STAGES) { stage = 0; phase ^= 1u; }
                        }
                        k += nb;
                    }
                    umma_commit(smem_u32(&sm->lo_full));
                    hi_phase ^= 1u;
                    lo_phase ^= 1u;
                }
                return true;
            };
            bool ok = true;
            for (int r = 0, t; ok && (t = round_tile(r)) < tiles && !*abort; ++r) {
                int m, n;
                map_tile(p, t, m, n);
                const int nk = tile_steps(m, n);
                for (int s0 = 0; s0 < nk && ok; s0 += SEG_STEPS)
                    ok = segment(min(SEG_STEPS, nk - s0));
            }
            // All MMAs issued by this CTA complete before TMEM is released.
            umma_commit(smem_u32(&sm->drain));
            wait(&sm->drain, 0, false);
        }
    } else {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(REGS_EPILOGUE));
        // ---------------- epilogue ----------------
        // warp w: TMEM lanes 32 (w % 4) .., columns [half * HC, half * HC + HC)
        constexpr int HC = BN / 2, W = HC < 16 ? HC : 16;
        const int q = warp & 3, half = (warp - 4) >> 2;
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
        bool ok = true;
        for (int r = 0, t; ok && (t = round_tile(r)) < tiles; ++r) {
            int m, n;
            map_tile(p, t, m, n);
            const int nkt = tile_steps(m, n);
            const int64_t row = (int64_t)m * BM + q * 32 + lane;
            const int64_t col0 = (int64_t)n * BN + half * HC;
            const bool row_ok = row < p.rows;
            const int64_t pieces = (int64_t)p.tn * 2;
            for (int seg = 0; seg * SEG_STEPS < nkt; ++seg) {
                const int nk = min(SEG_STEPS, nkt - seg * SEG_STEPS);
                const int2* qinfo = p.qinfo + seg * p.cols;
                const int2 ri = row_ok ? p.pinfo[seg * p.rows + row] : make_int2(0, 0);
                int bad = ri.x == kBadExp;
                if (!(ok = warp_wait(&sm->hi_full, hi_phase))) break;
                hi_phase ^= 1u;
#pragma unroll 1
                for (int c = 0; c < HC; c += 8) {
                    float v[8];
                    tmem_ld(tq + c, v);
                    tmem_wait_ld();
                    tmem_landed(v);
#pragma unroll
                    for (int u = 0; u < 8; ++u) {
                        if (col0 + c + u < p.cols && row_ok) {
                            const int2 ci = __ldg(qinfo + col0 + c + u);
                            const int cnt = min(ri.y, ci.y);
                            bad |= ci.x == kBadExp ||
                                   (cnt > 0 && !(v[u] >= (float)cnt * p.least));
                        }
                    }
                }
                release(&sm->hi_empty);
                bad = __any_sync(0xffffffffu, bad);
                // running sums: T in units of level 6, R in units of level 8. The
                // magic constant that turns level 2 into an integer comes off here,
                // once for all chunks.
                const long long nch = (nk + CHUNK - 1) / CHUNK;
                const long long t0 = -(nch * (0x4b400000ll << 32));
                long long T[HC];
                float R[HC];
#pragma unroll
                for (int c = 0; c < HC; ++c) {
                    T[c] = t0;
                    R[c] = 0.f;
                }
                for (int k0 = 0; k0 < nk; k0 += CHUNK) {
                    if (!(ok = warp_wait(&sm->hi_full, hi_phase))) break;
                    hi_phase ^= 1u;
#pragma unroll
                    for (int c = 0; c < HC; c += W) {
                        float l2[W], l3[W], l4[W], l5[W];
                        tmem_ld(tq + c, l2);
                        tmem_ld(tq + BN + c, l3);
                        tmem_ld(tq + 2 * BN + c, l4);
                        tmem_ld(tq + 3 * BN + c, l5);
                        tmem_wait_ld();
                        tmem_landed(l2);
                        tmem_landed(l3);
                        tmem_landed(l4);
                        tmem_landed(l5);
#pragma unroll
                        for (int u = 0; u < W; ++u) {
                            long long x = T[c + u];
                            x += (long long)__float2int_rn(l5[u]) << 8;
                            x += (long long)__float2int_rn(l4[u]) << 16;
                            x += (long long)__float2int_rn(l3[u]) << 24;
                            // |level 2| <= 192 * 2^14 < 2^22
                            x += (long long)((unsigned long long)__float_as_uint(l2[u] + kMagic) << 32);
                            T[c + u] = x;
                        }
                    }
                    release(&sm->hi_empty);
                    if (!(ok = warp_wait(&sm->lo_full, lo_phase))) break;
                    lo_phase ^= 1u;
#pragma unroll
                    for (int c = 0; c < HC; c += W) {
                        float l6[W], l7[W], l8[W], l9[W];
                        tmem_ld(tq + 4 * BN + c, l6);
                        tmem_ld(tq + 5 * BN + c, l7);
                        tmem_ld(tq + 6 * BN + c, l8);
                        tmem_ld(tq + 7 * BN + c, l9);
                        tmem_wait_ld();
                        tmem_landed(l6);
                        tmem_landed(l7);
                        tmem_landed(l8);
                        tmem_landed(l9);
#pragma unroll
                        for (int u = 0; u < W; ++u) {
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
                if (lane == 0 && row < p.rows && col0 < p.cols)
                    p.flags[seg * p.seg_flags + ((int64_t)m * 4 + q) * pieces + n * 2 + half] = bad;
                if (!row_ok || (bad && (seg > 0 || (p.E == p.D && p.c0 == 1.0 && !p.F)))) continue;
                // T 2^-48 + R 2^-64 as one double (units 2^-64), rounded once:
                // 2^100 + (T >> 32) 2^48 less its offset, plus the low 32 bits and
                // R in the mantissa of 2^52
                const double g = p.gamma * __hiloint2double((1023 + ri.x - 64) << 20, 0);
                double* dst = p.D + row * p.d_rs + col0 * p.d_cs;
                // the linear terms once, with the first segment
                const double* e = seg > 0 ? dst : p.E ? p.E + row * p.e_rs + col0 * p.e_cs : nullptr;
                const int64_t e_cs = seg > 0 ? p.d_cs : p.e_cs;
                const double c0 = seg > 0 ? 1.0 : p.c0;
                const double* f = seg > 0 || !p.F ? nullptr : p.F + row * p.f_rs + col0 * p.f_cs;
                double di = p.dg;
                if (f && p.tri == 1) di *= diagonal(p, row);
                // eight columns at a time: their loads all issued before the first
                // store (which may alias any later load for the compiler)
#pragma unroll
                for (int c8 = 0; c8 < HC; c8 += 8) {
                    double base[8];
                    int ce[8];
#pragma unroll
                    for (int u = 0; u < 8; ++u) {
                        const int c = c8 + u;
                        const bool in = col0 + c < p.cols;
                        base[u] = in && e ? __ldcg(e + c * e_cs) : 0.0;
                        ce[u] = in ? __ldg(qinfo + col0 + c).x : 0;
                    }
                    if (c0 != 1.0) {
#pragma unroll
                        for (int u = 0; u < 8; ++u) base[u] *= c0;
                    }
                    if (f) {
                        double fv[8];
#pragma unroll
                        for (int u = 0; u < 8; ++u)
                            fv[u] = col0 + c8 + u < p.cols ? __ldcg(f + (c8 + u) * p.f_cs) : 0.0;
#pragma unroll
                        for (int u = 0; u < 8; ++u) {
                            double d = di;
                            if (p.tri == 2)
                                d *= col0 + c8 + u < p.cols ? diagonal(p, col0 + c8 + u) : 0.0;
                            base[u] = fma(d, fv[u], base[u]);
                        }
                    }
#pragma unroll
                    for (int u = 0; u < 8; ++u) {
                        const int c = c8 + u;
                        const int th = (int)(T[c] >> 32);
                        const unsigned tl = (unsigned)T[c];
                        const double da = __hiloint2double(0x46300000, th ^ (int)0x80000000);
                        const unsigned long long mb =
                            0x4338000000000000ull + ((unsigned long long)tl << 16) +
                            (unsigned long long)(long long)__float2int_rn(R[c]);
                        const double v = (da - (0x1p100 + 0x1p79 + 0x1p52 + 0x1p51)) +
                                         __longlong_as_double((long long)mb);
                        // times 2^ce: v is zero or at least one
                        const int vh = __double2hiint(v);
                        const double vs = __hiloint2double(
                            (vh << 1) == 0 || bad ? 0 : vh + (ce[u] << 20),
                            bad ? 0 : __double2loint(v));
                        if (col0 + c < p.cols) dst[c * p.d_cs] = fma(g, vs, base[u]);
                    }
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

// Bytes of an operand's images (rows rounded up to its blocks; a triangle's
// blocks end with their last row) and of an update's scratch.
struct OperandBytes {
    size_t digits, mags, info;
};
static OperandBytes operand_bytes(int64_t rows, int64_t K, int br, bool tri) {
    const int64_t nk = (K + KS - 1) / KS, nb = (rows + br - 1) / br;
    const int64_t steps = steps_before(tri, br, nb, nk);
    OperandBytes o;
    o.mags = (size_t)up(steps * plane_bytes(br), 256);
    o.digits = o.mags * S;
    o.info = (size_t)up(nseg(K) * rows * (int64_t)sizeof(int2), 256);
    return o;
}
static size_t total(const OperandBytes& o) { return o.digits + o.mags + o.info; }
static size_t flag_bytes(int64_t rows, int64_t cols, int64_t K) {
    // pieces of 32 rows x at least 8 columns
    return (size_t)up(nseg(K) * (up(rows, BM) / 32) * (up(cols, 64) / 8) * (int64_t)sizeof(int),
                      256);
}
static unsigned char* place(Operand& o, unsigned char* at, const OperandBytes& b) {
    o.digits = at;
    o.mags = at + b.digits;
    o.info = reinterpret_cast<int2*>(at + b.digits + b.mags);
    return at + total(b);
}
template <typename T>
static Operand operand(const T* X, int64_t rs, int64_t ls, int64_t rows, int br, bool tri) {
    Operand o;
    o.X = X;
    o.rs = rs;
    o.ls = ls;
    o.rows = rows;
    o.br = br;
    o.tri = tri;
    o.digits = o.mags = nullptr;
    o.info = nullptr;
    o.copy = nullptr;
    return o;
}
// Tile width by the rounds of tiles per SM times a K step's clocks: the twelve
// MMAs of a step take 1184, 672 and 480 clocks at 64, 32 and 16 columns (measured
// per MMA: 40 clocks at N <= 32, N / 2 from 128 on), and the operands 768, 640
// and 576 at 64 bytes a clock.
static int tile_columns(int64_t rows, int64_t cols, int num_sms) {
    const int64_t tm = (rows + BM - 1) / BM;
    const auto cost = [&](int bn, int64_t step) {
        const int64_t tiles = tm * ((cols + bn - 1) / bn);
        return (tiles + num_sms - 1) / num_sms * step;
    };
    const int64_t c64 = cost(64, 1184), c32 = cost(32, 672), c16 = cost(16, 576);
    return c64 <= c32 && c64 <= c16 ? 64 : c32 <= c16 ? 32 : 16;
}

// Split both operands (o1 null: only the first).
template <typename T0>
static cudaError_t launch_split(const Operand& o0, const Operand* o1, int64_t K, cudaStream_t s) {
    SplitArgs a;
    a.op[0] = o0;
    a.op[1] = o1 ? *o1 : o0;
    a.K = K;
    a.nk = (int)((K + KS - 1) / KS);
    a.strips0 = (int)((o0.rows + STRIP - 1) / STRIP);
    const int64_t strips = a.strips0 + (o1 ? (o1->rows + STRIP - 1) / STRIP : 0);
    // few strips: several CTAs each, which all look for the exponent and share the digits
    // (256 columns with K 4096 55 -> 18 us; TRSM 1000 x 200 290 -> 285; more than 256
    // CTAs read more than they save: refined 4096 x 256 1351 us, with 1024 1367, 2048 1422)
    const int64_t parts = std::max<int64_t>(
        1, std::min({(int64_t)8, std::min<int64_t>(K, SEG) / 128, 256 / (strips * nseg(K))}));
    return launch_kernel(oz_split_kernel<T0>,
                         dim3((unsigned)strips, (unsigned)nseg(K), (unsigned)parts), dim3(SPLIT_NT),
                         0, s, a);
}

// The product of two split operands (the rest of `q` set by the caller), and
// the pieces it leaves out: gamma * sum of M (element (i, l) = Am[i*m_rs + l*m_cs])
// and Y added to D by the DFMA kernel.
template <typename TA>
static cudaError_t launch_product(Params& q, const Operand& a, const Operand& b, int64_t K,
                                  int* flags, const TA* Am, int64_t m_rs, int64_t m_cs,
                                  const double* Y, int64_t y_rs, int64_t y_cs, bool swap,
                                  int num_sms, cudaStream_t s) {
    const int bn = b.br;
    q.pd = a.digits;
    q.pm = a.mags;
    q.qd = b.digits;
    q.qm = b.mags;
    q.pinfo = a.info;
    q.qinfo = b.info;
    q.rows = a.rows;
    q.cols = b.rows;
    q.tri = a.tri ? 1 : b.tri ? 2 : 0;
    q.nk = (int)((K + KS - 1) / KS);
    q.tm = (int)((q.rows + BM - 1) / BM);
    q.tn = (int)((q.cols + bn - 1) / bn);
    const int across = q.tri == 2 ? q.tm : q.tn;
    q.band = q.tri == 0 ? 16 : across <= 16 ? 1 : across <= 32 ? 4 : 8;
    q.flags = flags;
    q.seg_flags = (int64_t)q.tm * 4 * q.tn * 2;
    const int64_t tiles = (int64_t)q.tm * q.tn;
    if (tiles > (int64_t)1 << 30) return cudaErrorInvalidValue;
    const dim3 grid((unsigned)std::min<int64_t>(tiles, num_sms));
    cudaError_t e =
        bn == 64   ? launch_kernel(oz_gemm_kernel<64>, grid, dim3(NT), Cfg<64>::SMEM_BYTES, s, q)
        : bn == 32 ? launch_kernel(oz_gemm_kernel<32>, grid, dim3(NT), Cfg<32>::SMEM_BYTES, s, q)
                   : launch_kernel(oz_gemm_kernel<16>, grid, dim3(NT), Cfg<16>::SMEM_BYTES, s, q);
    if (e != cudaSuccess) return e;
    OzPieces pc;
    pc.flags = flags;
    pc.per_row = (int64_t)q.tn * 2;
    pc.per_seg = q.seg_flags;
    pc.cols = bn / 2;
    pc.seg = SEG;
    pc.swap = swap;
    pc.tri = q.tri != 0;
    return launch_gemm_simt_pieces(Am, m_rs, m_cs, swap ? q.cols : q.rows, K, Y, y_rs, y_cs,
                                   swap ? q.rows : q.cols, q.gamma, q.D, swap ? q.d_cs : q.d_rs,
                                   swap ? q.d_rs : q.d_cs, pc, s, num_sms);
}

static Params params(double gamma, float least, int* err, long long wait_ns) {
    Params q;
    q.E = q.F = nullptr;
    q.e_rs = q.e_cs = q.f_rs = q.f_cs = q.d_step = 0;
    q.c0 = 1.0;
    q.dg = 0.0;
    q.diag = nullptr;
    q.diag_f32 = 0;
    q.gamma = gamma;
    q.least = least;
    q.err = err;
    q.wait_ns = wait_ns;
    return q;
}
constexpr float kLeastFp64 = 0x1p-12f, kLeastResidual = 0x1p-16f;

// Tile rows (TMEM lanes) lie along C's contiguous index: the epilogue's lanes
// then read and write whole lines of C.
template <typename T>
static bool rows_are_rhs(const Canon<T>& p) {
    return (p.c_cs == 1 || p.c_cs == -1) && p.c_rs != 1 && p.c_rs != -1;
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

// Scratch: both operands in either orientation, whatever the tile width.
static size_t oz_bytes(int64_t rows, int64_t nrhs, int64_t K, bool tri) {
    using namespace oz;
    size_t most = 0;
    for (int swap = 0; swap < 2; ++swap)
        for (int bn = 16; bn <= 64; bn *= 2) {
            const size_t m = total(operand_bytes(rows, K, swap ? bn : BM, tri));
            const size_t y = total(operand_bytes(nrhs, K, swap ? BM : bn, false));
            most = std::max(most, m + y + flag_bytes(swap ? nrhs : rows, swap ? rows : nrhs, K));
        }
    return most;
}
size_t oz_update_bytes(int64_t mlen, int64_t nrhs, int64_t klen) {
    return oz_bytes(mlen, nrhs, klen, false);
}

cudaError_t launch_oz_update(const Canon<double>& p, const TcGemm& g, double beta, double gamma,
                             void* ws, int* err, long long wait_ns, int num_sms, cudaStream_t s) {
    using namespace oz;
    const bool swap = rows_are_rhs(p);
    const int64_t rows = swap ? p.nrhs : g.mlen, cols = swap ? g.mlen : p.nrhs;
    const int bn = tile_columns(rows, cols, num_sms);
    const double* M = p.A + g.rc * p.a_rs + g.rk * p.a_cs;
    const double* Y = p.C + g.rk * p.c_rs;
    Operand m = operand(M, p.a_rs, p.a_cs, g.mlen, swap ? bn : BM, false);
    Operand y = operand(Y, p.c_cs, p.c_rs, p.nrhs, swap ? BM : bn, false);
    unsigned char* at = place(m, static_cast<unsigned char*>(ws),
                              operand_bytes(g.mlen, g.klen, m.br, false));
    at = place(y, at, operand_bytes(p.nrhs, g.klen, y.br, false));
    const Operand &a = swap ? y : m, &b = swap ? m : y;
    cudaError_t e = launch_split<double>(a, &b, g.klen, s);
    if (e != cudaSuccess) return e;
    Params q = params(gamma, kLeastFp64, err, wait_ns);
    q.D = p.C + g.rc * p.c_rs;
    q.d_rs = swap ? p.c_cs : p.c_rs;
    q.d_cs = swap ? p.c_rs : p.c_cs;
    q.E = q.D;
    q.e_rs = q.d_rs;
    q.e_cs = q.d_cs;
    q.c0 = beta;
    return launch_product(q, a, b, g.klen, reinterpret_cast<int*>(at), M, p.a_rs, p.a_cs, Y,
                          p.c_rs, p.c_cs, swap, num_sms, s);
}

size_t oz_trmm_bytes(int64_t k, int64_t nrhs) {
    return oz_bytes(k, nrhs, k, true) + (size_t)oz::up(k * nrhs * 8, 256);
}

// C := alpha M C, M's strictly lower part on the tensor cores and its diagonal
// in the epilogue, from C's own element. The original right-hand side is in
// the digits, and copied for the DFMA pieces.
cudaError_t launch_oz_trmm(const Canon<double>& p, double alpha, void* ws, int* err,
                           long long wait_ns, int num_sms, cudaStream_t s) {
    using namespace oz;
    const bool swap = rows_are_rhs(p);
    const int bn = tile_columns(swap ? p.nrhs : p.k, swap ? p.k : p.nrhs, num_sms);
    Operand m = operand(p.A, p.a_rs, p.a_cs, p.k, swap ? bn : BM, true);
    Operand y = operand<double>(p.C, p.c_cs, p.c_rs, p.nrhs, swap ? BM : bn, false);
    unsigned char* at = static_cast<unsigned char*>(ws);
    y.copy = reinterpret_cast<double*>(at);
    at = place(m, at + up(p.k * p.nrhs * 8, 256), operand_bytes(p.k, p.k, m.br, true));
    at = place(y, at, operand_bytes(p.nrhs, p.k, y.br, false));
    const Operand &a = swap ? y : m, &b = swap ? m : y;
    cudaError_t e = launch_split<double>(a, &b, p.k, s);
    if (e != cudaSuccess) return e;
    Params q = params(alpha, kLeastFp64, err, wait_ns);
    q.D = p.C;
    q.d_rs = swap ? p.c_cs : p.c_rs;
    q.d_cs = swap ? p.c_rs : p.c_cs;
    q.F = q.D;
    q.f_rs = q.d_rs;
    q.f_cs = q.d_cs;
    q.dg = alpha;
    q.diag = p.unit ? nullptr : p.A;
    q.d_step = p.a_rs + p.a_cs;
    return launch_product(q, a, b, p.k, reinterpret_cast<int*>(at), p.A, p.a_rs, p.a_cs, y.copy,
                          1, p.k, swap, num_sms, s);
}

// The residual R := B - M X of the canonical k x k triangle (FP32 or FP64 data),
// M split once (oz_residual_split_m) for all the corrections that follow.
size_t oz_residual_bytes(int64_t k, int64_t n) { return oz_bytes(k, n, k, true); }

template <typename T>
static oz::Operand residual_m(const Canon<T>& p, void* ws, unsigned char** rest) {
    using namespace oz;
    Operand m = operand(p.A, p.a_rs, p.a_cs, p.k, BM, true);
    *rest = place(m, static_cast<unsigned char*>(ws), operand_bytes(p.k, p.k, BM, true));
    return m;
}
template <typename T>
cudaError_t oz_residual_split_m(const Canon<T>& p, void* ws, cudaStream_t s) {
    unsigned char* rest;
    return oz::launch_split<T>(residual_m(p, ws, &rest), nullptr, p.k, s);
}
template <typename T>
cudaError_t launch_oz_residual(const Canon<T>& p, const double* X, const double* B, double* R,
                               int64_t c_rs, int64_t c_cs, void* ws, int* err, long long wait_ns,
                               int num_sms, cudaStream_t s) {
    using namespace oz;
    unsigned char* at;
    const Operand m = residual_m(p, ws, &at);
    Operand x = operand(X, c_cs, c_rs, p.nrhs, tile_columns(p.k, p.nrhs, num_sms), false);
    at = place(x, at, operand_bytes(p.nrhs, p.k, x.br, false));
    cudaError_t e = launch_split<double>(x, nullptr, p.k, s);
    if (e != cudaSuccess) return e;
    Params q = params(-1.0, kLeastResidual, err, wait_ns);
    q.D = R;
    q.E = B;
    q.F = X;
    q.d_rs = q.e_rs = q.f_rs = c_rs;
    q.d_cs = q.e_cs = q.f_cs = c_cs;
    q.dg = -1.0;
    q.diag = p.unit ? nullptr : p.A;
    q.diag_f32 = sizeof(T) == 4;
    q.d_step = p.a_rs + p.a_cs;
    return launch_product(q, m, x, p.k, reinterpret_cast<int*>(at), p.A, p.a_rs, p.a_cs, X, c_rs,
                          c_cs, false, num_sms, s);
}
template cudaError_t oz_residual_split_m<float>(const Canon<float>&, void*, cudaStream_t);
template cudaError_t oz_residual_split_m<double>(const Canon<double>&, void*, cudaStream_t);
template cudaError_t launch_oz_residual<float>(const Canon<float>&, const double*, const double*,
                                               double*, int64_t, int64_t, void*, int*, long long,
                                               int, cudaStream_t);
template cudaError_t launch_oz_residual<double>(const Canon<double>&, const double*,
                                                const double*, double*, int64_t, int64_t, void*,
                                                int*, long long, int, cudaStream_t);

}  // namespace trx
