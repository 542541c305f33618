// CUDA-core GEMM update (FP32 FMA / FP64 DFMA) on the canonical matrices:
//
//   C[rc+i, j] = beta * C[rc+i, j] + gamma * sum_l M(rc+i, rk+l) * Y[rk+l, j]
//
// with Y = C (a different row block of the same buffer) inside the recursion.
// This is the off-diagonal step of the recursion (Section 3.1): for TRSM
// B2 := beta*B2 - M21 X1 (gamma = -1), for TRMM B2 += alpha M21 B1. Rows
// [rc, rc+mlen) and [rk, rk+klen) are disjoint row blocks of one buffer.
//
// It is the GEMM engine of the FP64 path (tcgen05 has no FP64 kind), the
// FP32 path's engine for small updates whose K is not a multiple of the
// tensor-core K tile, and the FP32 engine when the tensor cores are switched
// off. Tile 64x64x16, 256 threads, 4x4 outputs per thread, operands staged
// through shared memory with the global loop order chosen so the contiguous
// index runs fastest (the matrices arrive with arbitrary signed strides).
// An update with fewer 64x64 tiles than twice the SMs takes 32x32 (2x2
// outputs per thread) or 16x16 tiles (one output), four or sixteen times the
// CTAs: the FP64 pipe is about 1/64 of the FP32 one per SM on this part, so
// a small FP64 update on a few SMs was the FP64 path's bottleneck at small
// orders.
#include <type_traits>

#include "common.cuh"

namespace trx {
namespace {

constexpr int BK = 16, NT = 256;

template <typename T>
struct GemmArgs {
    Canon<T> p;
    const T* Y;            // K operand, Y(l, j) = Y[l*y_rs + j*y_cs] (C in the recursion)
    int64_t y_rs, y_cs;
    int64_t rc, mlen, rk, klen;
    T beta, gamma;
};

// TM x TM outputs per thread; tile BM = BN = 16 TM.
template <typename T, int TM>
__global__ void __launch_bounds__(NT) gemm_simt_kernel(GemmArgs<T> g) {
    constexpr int BM = 16 * TM, BN = 16 * TM, LE = BM * BK / NT;   // loads per thread
    __shared__ T sA[2][BK][BM + 4];   // sA[l][i] = M(rc+i0+i, rk+l0+l)
    __shared__ T sB[2][BK][BN + 4];   // sB[l][j] = C(rk+l0+l, j0+j)
    pdl_trigger();
    pdl_wait();
    const Canon<T>& p = g.p;
    const int tid = threadIdx.x;
    const int tx = tid % 16, ty = tid / 16;
    const int64_t i0 = (int64_t)blockIdx.y * BM;
    const int64_t j0 = (int64_t)blockIdx.x * BN;
    const bool a_row_fast = (p.a_rs == 1 || p.a_rs == -1);
    const bool y_row_fast = (g.y_rs == 1 || g.y_rs == -1);

    T ra[LE], rb[LE];
    auto load = [&](int64_t l0) {
#pragma unroll
        for (int u = 0; u < LE; ++u) {
            const int e = tid + u * NT;
            int i, l;
            if (a_row_fast) { i = e % BM; l = e / BM; } else { l = e % BK; i = e / BK; }
            const int64_t gi = i0 + i, gl = l0 + l;
            ra[u] = (gi < g.mlen && gl < g.klen) ? p.A[(g.rc + gi) * p.a_rs + (g.rk + gl) * p.a_cs] : T(0);
            int lb, jb;
            if (y_row_fast) { lb = e % BK; jb = e / BK; } else { jb = e % BN; lb = e / BN; }
            const int64_t gl2 = l0 + lb, gj = j0 + jb;
            rb[u] = (gl2 < g.klen && gj < p.nrhs) ? g.Y[(g.rk + gl2) * g.y_rs + gj * g.y_cs] : T(0);
        }
    };
    auto store = [&](int buf) {
#pragma unroll
        for (int u = 0; u < LE; ++u) {
            const int e = tid + u * NT;
            int i, l;
            if (a_row_fast) { i = e % BM; l = e / BM; } else { l = e % BK; i = e / BK; }
            sA[buf][l][i] = ra[u];
            int lb, jb;
            if (y_row_fast) { lb = e % BK; jb = e / BK; } else { jb = e % BN; lb = e / BN; }
            sB[buf][lb][jb] = rb[u];
        }
    };

    T acc[TM][TM];
#pragma unroll
    for (int u = 0; u < TM; ++u)
#pragma unroll
        for (int v = 0; v < TM; ++v) acc[u][v] = T(0);

    int buf = 0;
    load(0);
    store(0);
    __syncthreads();
    for (int64_t l0 = 0; l0 < g.klen; l0 += BK) {
        const bool more = l0 + BK < g.klen;
        if (more) load(l0 + BK);   // next tile in flight during the FMAs
#pragma unroll
        for (int l = 0; l < BK; ++l) {
            T a[TM], b[TM];
#pragma unroll
            for (int u = 0; u < TM; ++u) a[u] = sA[buf][l][tx + 16 * u];
#pragma unroll
            for (int v = 0; v < TM; ++v) b[v] = sB[buf][l][ty + 16 * v];
#pragma unroll
            for (int u = 0; u < TM; ++u)
#pragma unroll
                for (int v = 0; v < TM; ++v) acc[u][v] = fma(a[u], b[v], acc[u][v]);
        }
        if (more) {
            store(buf ^ 1);
            __syncthreads();
            buf ^= 1;
        }
    }
#pragma unroll
    for (int u = 0; u < TM; ++u) {
        const int64_t gi = i0 + tx + 16 * u;
        if (gi >= g.mlen) continue;
#pragma unroll
        for (int v = 0; v < TM; ++v) {
            const int64_t gj = j0 + ty + 16 * v;
            if (gj >= p.nrhs) continue;
            T* c = p.C + (g.rc + gi) * p.c_rs + gj * p.c_cs;
            *c = g.beta * *c + g.gamma * acc[u][v];
        }
    }
}

template <typename TA>
struct PieceArgs {
    const TA* A;           // A(i, l) = A[i*a_rs + l*a_cs]
    int64_t a_rs, a_cs, mlen, klen;
    const double* Y;       // Y(l, j) = Y[l*y_rs + j*y_cs]
    int64_t y_rs, y_cs, nrhs;
    double gamma;
    double* D;             // D(i, j) = D[i*d_rs + j*d_cs]
    int64_t d_rs, d_cs;
    OzPieces pc;
};

// The DFMA update over the pieces that the tensor-core update (gemm_oz.cu) left
// out, D(i, j) += gamma * sum_l A(i, l) Y(l, j) segment by segment of l, same
// tiles as above. A tile without a flag only reads its flags (3 us for a
// 2048 x 4096 update).
template <typename TA, int TM>
__global__ void __launch_bounds__(NT, 2) gemm_pieces_kernel(PieceArgs<TA> g) {
    constexpr int BM = 16 * TM, BN = 16 * TM, LE = BM * BK / NT;
    __shared__ double sA[2][BK][BM + 4];
    __shared__ double sB[2][BK][BN + 4];
    pdl_trigger();
    pdl_wait();
    const int tid = threadIdx.x;
    const int tx = tid % 16, ty = tid / 16;
    const int64_t i0 = (int64_t)blockIdx.y * BM, j0 = (int64_t)blockIdx.x * BN;
    const bool a_row_fast = (g.a_rs == 1 || g.a_rs == -1);
    const bool y_row_fast = (g.y_rs == 1 || g.y_rs == -1);
    const int64_t kmax = g.pc.tri ? min(g.klen, i0 + BM) : g.klen;
    for (int seg = 0; (int64_t)seg * g.pc.seg < kmax; ++seg) {
        const int64_t k0 = (int64_t)seg * g.pc.seg, k1 = min(kmax, k0 + g.pc.seg);
        const int* flags = g.pc.flags + seg * g.pc.per_seg;
        const auto flagged = [&](int64_t i, int64_t j) {
            if (g.pc.tri && k0 >= i) return 0;           // no terms (and no flag) there
            const int64_t r = g.pc.swap ? j : i, c = g.pc.swap ? i : j;
            return flags[(r >> 5) * g.pc.per_row + c / g.pc.cols];
        };
        // the tile's flags, at the granularity of the smallest piece (8); the
        // last row of eight has terms where any of them has
        int any = 0;
        for (int e = tid; e < (BM / 8) * (BN / 8); e += NT) {
            const int64_t i = i0 + e / (BN / 8) * 8, j = j0 + e % (BN / 8) * 8;
            if (i < g.mlen && j < g.nrhs) any |= flagged(min(i + 7, g.mlen - 1), j);
        }
        if (!__syncthreads_or(any)) continue;
        double ra[LE], rb[LE];
        auto load = [&](int64_t l0) {
#pragma unroll
            for (int u = 0; u < LE; ++u) {
                const int e = tid + u * NT;
                const int i = a_row_fast ? e % BM : e / BK, l = a_row_fast ? e / BM : e % BK;
                const int64_t gi = i0 + i, gl = l0 + l;
                ra[u] = (gi < g.mlen && gl < (g.pc.tri ? min(k1, gi) : k1))
                            ? (double)g.A[gi * g.a_rs + gl * g.a_cs]
                            : 0.0;
                const int lb = y_row_fast ? e % BK : e / BN, jb = y_row_fast ? e / BK : e % BN;
                const int64_t gl2 = l0 + lb, gj = j0 + jb;
                rb[u] = (gl2 < k1 && gj < g.nrhs) ? g.Y[gl2 * g.y_rs + gj * g.y_cs] : 0.0;
            }
        };
        auto store = [&](int buf) {
#pragma unroll
            for (int u = 0; u < LE; ++u) {
                const int e = tid + u * NT;
                sA[buf][a_row_fast ? e / BM : e % BK][a_row_fast ? e % BM : e / BK] = ra[u];
                sB[buf][y_row_fast ? e % BK : e / BN][y_row_fast ? e / BK : e % BN] = rb[u];
            }
        };
        double acc[TM][TM];
#pragma unroll
        for (int u = 0; u < TM; ++u)
#pragma unroll
            for (int v = 0; v < TM; ++v) acc[u][v] = 0.0;
        int buf = 0;
        load(k0);
        store(0);
        __syncthreads();
        for (int64_t l0 = k0; l0 < k1; l0 += BK) {
            const bool more = l0 + BK < k1;
            if (more) load(l0 + BK);
            // a triangle's steps at its diagonal: a row takes part only in the products
            // left of it (a zero in A's place times an Inf or NaN of Y would be a NaN)
            const auto products = [&](auto edge) {
#pragma unroll
                for (int l = 0; l < BK; ++l) {
                    double a[TM], b[TM];
#pragma unroll
                    for (int u = 0; u < TM; ++u) a[u] = sA[buf][l][tx + 16 * u];
#pragma unroll
                    for (int v = 0; v < TM; ++v) b[v] = sB[buf][l][ty + 16 * v];
#pragma unroll
                    for (int u = 0; u < TM; ++u) {
                        if (decltype(edge)::value && l0 + l >= i0 + tx + 16 * u) continue;
#pragma unroll
                        for (int v = 0; v < TM; ++v) acc[u][v] = fma(a[u], b[v], acc[u][v]);
                    }
                }
            };
            if (g.pc.tri && l0 + BK > i0) products(std::true_type{});
            else products(std::false_type{});
            if (more) {
                store(buf ^ 1);
                __syncthreads();
                buf ^= 1;
            }
        }
#pragma unroll
        for (int u = 0; u < TM; ++u) {
            const int64_t gi = i0 + tx + 16 * u;
            if (gi >= g.mlen) continue;
#pragma unroll
            for (int v = 0; v < TM; ++v) {
                const int64_t gj = j0 + ty + 16 * v;
                if (gj >= g.nrhs || !flagged(gi, gj)) continue;
                double* d = g.D + gi * g.d_rs + gj * g.d_cs;
                *d = fma(g.gamma, acc[u][v], *d);
            }
        }
        __syncthreads();                     // sA and sB are refilled
    }
}

// The largest tile (64, 32, 16 rows) that still gives every SM two CTAs.
int tile_factor(int64_t rows, int64_t cols, int num_sms) {
    const auto tiles = [&](int tm) {
        return ((rows + 16 * tm - 1) / (16 * tm)) * ((cols + 16 * tm - 1) / (16 * tm));
    };
    const int64_t want = 2 * (int64_t)(num_sms > 0 ? num_sms : 1);
    return tiles(4) >= want ? 4 : tiles(2) >= want ? 2 : 1;
}

}  // namespace

template <typename T>
cudaError_t launch_gemm_simt(const Canon<T>& p, const T* Y, int64_t y_rs, int64_t y_cs,
                             int64_t rc, int64_t mlen, int64_t rk, int64_t klen, T beta,
                             T gamma, cudaStream_t s, int num_sms) {
    if (mlen <= 0 || p.nrhs <= 0) return cudaSuccess;
    GemmArgs<T> g;
    g.p = p;
    g.Y = Y;
    g.y_rs = y_rs;
    g.y_cs = y_cs;
    g.rc = rc;
    g.mlen = mlen;
    g.rk = rk;
    g.klen = klen;
    g.beta = beta;
    g.gamma = gamma;
    const int tm = tile_factor(mlen, p.nrhs, num_sms);
    const int64_t gy = (mlen + 16 * tm - 1) / (16 * tm), gx = (p.nrhs + 16 * tm - 1) / (16 * tm);
    if (gy > 65535) return cudaErrorInvalidValue;
    const dim3 grid((unsigned)gx, (unsigned)gy);
    if (tm == 1) return launch_kernel(gemm_simt_kernel<T, 1>, grid, dim3(NT), 0, s, g);
    if (tm == 2) return launch_kernel(gemm_simt_kernel<T, 2>, grid, dim3(NT), 0, s, g);
    return launch_kernel(gemm_simt_kernel<T, 4>, grid, dim3(NT), 0, s, g);
}

template <typename TA>
cudaError_t launch_gemm_simt_pieces(const TA* A, int64_t a_rs, int64_t a_cs, int64_t mlen,
                                    int64_t klen, const double* Y, int64_t y_rs, int64_t y_cs,
                                    int64_t nrhs, double gamma, double* D, int64_t d_rs,
                                    int64_t d_cs, const OzPieces& pieces, cudaStream_t s,
                                    int num_sms) {
    PieceArgs<TA> g;
    g.A = A;
    g.a_rs = a_rs;
    g.a_cs = a_cs;
    g.mlen = mlen;
    g.klen = klen;
    g.Y = Y;
    g.y_rs = y_rs;
    g.y_cs = y_cs;
    g.nrhs = nrhs;
    g.gamma = gamma;
    g.D = D;
    g.d_rs = d_rs;
    g.d_cs = d_cs;
    g.pc = pieces;
    const int tm = tile_factor(mlen, nrhs, num_sms);
    const int64_t gy = (mlen + 16 * tm - 1) / (16 * tm), gx = (nrhs + 16 * tm - 1) / (16 * tm);
    if (gy > 65535) return cudaErrorInvalidValue;
    const dim3 grid((unsigned)gx, (unsigned)gy);
    // its launch overlaps the tensor-core update's tail (it waits for that kernel
    // before it reads a flag): 2 us less an update. The same on the update itself,
    // over the operand split, gained 3 us alone and lost 1-2 % inside launch graphs.
    const PdlScope overlap;
    if (tm == 1) return launch_kernel(gemm_pieces_kernel<TA, 1>, grid, dim3(NT), 0, s, g);
    if (tm == 2) return launch_kernel(gemm_pieces_kernel<TA, 2>, grid, dim3(NT), 0, s, g);
    return launch_kernel(gemm_pieces_kernel<TA, 4>, grid, dim3(NT), 0, s, g);
}
template cudaError_t launch_gemm_simt_pieces<float>(const float*, int64_t, int64_t, int64_t,
                                                    int64_t, const double*, int64_t, int64_t,
                                                    int64_t, double, double*, int64_t, int64_t,
                                                    const OzPieces&, cudaStream_t, int);
template cudaError_t launch_gemm_simt_pieces<double>(const double*, int64_t, int64_t, int64_t,
                                                     int64_t, const double*, int64_t, int64_t,
                                                     int64_t, double, double*, int64_t, int64_t,
                                                     const OzPieces&, cudaStream_t, int);

template cudaError_t launch_gemm_simt<float>(const Canon<float>&, const float*, int64_t, int64_t,
                                             int64_t, int64_t, int64_t, int64_t, float, float,
                                             cudaStream_t, int);
template cudaError_t launch_gemm_simt<double>(const Canon<double>&, const double*, int64_t,
                                              int64_t, int64_t, int64_t, int64_t, int64_t,
                                              double, double, cudaStream_t, int);

}  // namespace trx
