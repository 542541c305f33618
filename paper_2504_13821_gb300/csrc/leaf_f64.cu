// FP64 TRSM leaves (Section 3.3 base kernel). First, 33..64 rows with many right-hand
// sides: blocked forward substitution in 16-row blocks, C columns per CTA of 128
// threads.
//
// The FP64 pipe takes two FMAs per clock and SM: one FP64 instruction of a warp
// holds it for 16 clocks, however few of its lanes count, and the substitution is
// a chain of 64 multiply / FMA pairs. So L = 128 / C lanes share a column there (16 /
// L rows each, x_j by shuffle), which keeps every lane's part of the chain short,
// and in the rank-16 updates below the block every thread owns the same number of
// rows x columns. Tiles are narrow (8 columns up to 8 an SM, 16 beyond) so that
// every SM has one and two or three overlap one another's chains; the kernel of 64
// columns per CTA and one lane per column that this one replaces kept 64 SMs busy
// at 4096 right-hand sides.
//
// Measured, one 64-row leaf (us by right-hand sides, that kernel / this one, ncu):
// 1024 47 / 17, 1500 48 / 21, 4096 54 / 29 (30 with the products summed first); four lanes per column took 20 (1024)
// and 29 (4096), 32 columns per CTA 34 (4096). Up to 1024 right-hand sides
// leaf256_kernel below serves.
#include "common.cuh"
#include "leaf_impl.cuh"

namespace trx {
namespace {

template <int C>
struct Leaf64 {
    static constexpr int NT = 128, B = 64, SB = 16;
    static constexpr int L = NT / C;                 // lanes per column in the substitution
    static constexpr int RU = SB / L;                // rows per lane
    static constexpr int CW = C / 8;   // columns per thread in the updates
    static constexpr int CG = C / CW, RG = NT / CG;  // column and row groups
    static constexpr int LDT = B + 1;                // column stride of the triangle
    static constexpr int LDC = C + 2;                // row stride of the panel
    static constexpr size_t smem = sizeof(double) * (size_t)(B * LDT + B + B * LDC);
    static_assert(RG == SB, "a block's rows below divide evenly over the row groups");
};

template <int C>
__global__ void __launch_bounds__(128) leaf64_kernel(LeafArgs<double> a) {
    using S = Leaf64<C>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    double* sT = reinterpret_cast<double*>(smem_raw);    // M(r0+i, r0+l) at l*LDT + i, i > l
    double* sD = sT + S::B * S::LDT;                       // reciprocal diagonal
    double* sC = sD + S::B;                                // C(r0+i, j0+c) at i*LDC + c
    pdl_trigger();
    pdl_wait();
    const int tid = threadIdx.x;
    const Canon<double>& p = a.p;
    const int64_t r0 = a.r0, j0 = (int64_t)blockIdx.x * C;
    const int bs = (int)min((int64_t)a.b, p.k - r0);
    const int nc = (int)min((int64_t)C, p.nrhs - j0);

    // panel and triangle along their contiguous index, every load of the panel
    // in flight at once; rows past the leaf and columns past C are zero
    constexpr int PL = S::B * C / S::NT;
    const bool c_row_fast = p.c_rs == 1 || p.c_rs == -1;
    double v[PL];
#pragma unroll
    for (int u = 0; u < PL; ++u) {
        const int e = tid + u * S::NT;
        const int i = c_row_fast ? e % S::B : e / C, c = c_row_fast ? e / S::B : e % C;
        v[u] = i < bs && c < nc ? p.C[(r0 + i) * p.c_rs + (j0 + c) * p.c_cs] : 0.0;
    }
    const bool a_row_fast = p.a_rs == 1 || p.a_rs == -1;
    const double* A = p.A + r0 * (p.a_rs + p.a_cs);
    constexpr int TL = S::B * S::B / S::NT;
    double d = 1.0;
    if (tid < bs && !p.unit) d = A[tid * (p.a_rs + p.a_cs)];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        double t[TL / 2];
#pragma unroll
        for (int u = 0; u < TL / 2; ++u) {
            const int e = tid + (h * (TL / 2) + u) * S::NT;
            const int i = a_row_fast ? e % S::B : e / S::B, l = a_row_fast ? e / S::B : e % S::B;
            t[u] = l < i && i < bs ? A[i * p.a_rs + l * p.a_cs] : 0.0;
        }
#pragma unroll
        for (int u = 0; u < TL / 2; ++u) {
            const int e = tid + (h * (TL / 2) + u) * S::NT;
            const int i = a_row_fast ? e % S::B : e / S::B, l = a_row_fast ? e / S::B : e % S::B;
            sT[l * S::LDT + i] = t[u];
        }
    }
    if (tid < S::B) sD[tid] = 1.0 / d;
#pragma unroll
    for (int u = 0; u < PL; ++u) {
        const int e = tid + u * S::NT;
        const int i = c_row_fast ? e % S::B : e / C, c = c_row_fast ? e / S::B : e % C;
        sC[i * S::LDC + c] = a.alpha * v[u];
    }
    __syncthreads();

    const int sc = tid / S::L, sg = tid % S::L;            // substitution: column, lane of it
    const int cg = tid % S::CG, rg = tid / S::CG;          // updates: columns, rows
#pragma unroll
    for (int s0 = 0; s0 < S::B; s0 += S::SB) {
        // rows s0 .. s0+15 of column sc: lane sg holds rows sg + L u
        double x[S::RU];
#pragma unroll
        for (int u = 0; u < S::RU; ++u) x[u] = sC[(s0 + sg + S::L * u) * S::LDC + sc];
#pragma unroll
        for (int j = 0; j < S::SB; ++j) {
            const double xj = __shfl_sync(0xffffffffu, x[j / S::L], j % S::L, S::L) * sD[s0 + j];
            if (sg == j % S::L) x[j / S::L] = xj;
#pragma unroll
            for (int u = j / S::L; u < S::RU; ++u) {
                const int i = sg + S::L * u;
                if (i > j) x[u] = fma(-sT[(s0 + j) * S::LDT + s0 + i], xj, x[u]);
            }
        }
#pragma unroll
        for (int u = 0; u < S::RU; ++u) sC[(s0 + sg + S::L * u) * S::LDC + sc] = x[u];
        __syncthreads();
        // rank-16 update of the rows below: the 16 products are summed before they meet
        // the row, whose roundings stay as few as an update's between leaves
        constexpr int UMAX = S::B / S::SB - 1;
        const int nu = UMAX - s0 / S::SB;                  // compile-time after unrolling
        double acc[UMAX][S::CW] = {};
#pragma unroll
        for (int kk = 0; kk < S::SB; ++kk) {
            double xv[S::CW];
#pragma unroll
            for (int w = 0; w < S::CW; ++w) xv[w] = sC[(s0 + kk) * S::LDC + cg * S::CW + w];
#pragma unroll
            for (int u = 0; u < UMAX; ++u) {
                if (u >= nu) continue;
                const double t = sT[(s0 + kk) * S::LDT + s0 + S::SB * (u + 1) + rg];
#pragma unroll
                for (int w = 0; w < S::CW; ++w) acc[u][w] = fma(-t, xv[w], acc[u][w]);
            }
        }
#pragma unroll
        for (int u = 0; u < UMAX; ++u)
#pragma unroll
            for (int w = 0; w < S::CW; ++w)
                if (u < nu) sC[(s0 + S::SB * (u + 1) + rg) * S::LDC + cg * S::CW + w] += acc[u][w];
        __syncthreads();
    }
#pragma unroll
    for (int u = 0; u < PL; ++u) {
        const int e = tid + u * S::NT;
        const int i = c_row_fast ? e % S::B : e / C, c = c_row_fast ? e / S::B : e % C;
        if (i < bs && c < nc) p.C[(r0 + i) * p.c_rs + (j0 + c) * p.c_cs] = sC[i * S::LDC + c];
    }
}

// FP64 TRSM leaf of 33..256 rows with few right-hand sides, C columns a CTA, in 16-row
// blocks: warp 0 substitutes block q (32 / C lanes a column) while warps 1-3 take block
// q - 1's columns off the rows below it and four more warps bring M's columns of block
// q + 1 in; then the four take block q's columns off block q + 1.
//
// Bound by the chain: an FP64 instruction holds its warp's quarter of the pipe for 64
// clocks, so a step (shuffle, multiply, FMA) takes about 200 and the rows below must be
// other warps' work. Leaves of 64 rows have the same chain and, every 64 rows, a
// launch and an update that 200 right-hand sides cannot spread over the SMs.
// A TRSM of order 1000 with 200 right-hand sides: leaves of 64 rows 395 us, a warp a
// column with all its rows in the one warp 400, this kernel 280.
template <int C>
struct Leaf256 {
    static constexpr int NT = 256, B = 256, SB = 16, STAGES = 3;
    static constexpr int LDT = B + 1;                // column stride: transposed copies, 32 banks
    static constexpr int L = 32 / C;                 // lanes a column in the substitution
    static constexpr int RU = SB / L;                // rows a lane
    static constexpr int KS = 128 / (SB * C);        // lanes an element in the next block's update
    static constexpr size_t smem = sizeof(double) * (size_t)(STAGES * SB * LDT + B + B * C);
};

__device__ __forceinline__ void cp_async8(double* dst, const double* src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(
                     (uint32_t)__cvta_generic_to_shared(dst)),
                 "l"(src)
                 : "memory");
}

template <int C>
__global__ void __launch_bounds__(256) leaf256_kernel(LeafArgs<double> a) {
    using S = Leaf256<C>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    double* sP = reinterpret_cast<double*>(smem_raw);   // M(r0+i, r0+16q+l) at l*LDT + i, i below
    double* sD = sP + S::STAGES * S::SB * S::LDT;         // reciprocal diagonal
    double* sC = sD + S::B;                                // C(r0+i, j0+c) at i*C + c
    pdl_trigger();
    pdl_wait();
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const Canon<double>& p = a.p;
    const int64_t r0 = a.r0, j0 = (int64_t)blockIdx.x * C;
    const int bs = (int)min((int64_t)a.b, p.k - r0);
    const int nq = (bs + S::SB - 1) / S::SB;
    const int nc = (int)min((int64_t)C, p.nrhs - j0);
    const double* A = p.A + r0 * (p.a_rs + p.a_cs);
    double* Cp = p.C + r0 * p.c_rs + j0 * p.c_cs;

    const auto panel = [&](int q) { return sP + q % S::STAGES * S::SB * S::LDT; };
    const auto load = [&](int q) {   // warps 4-7
        double* dst = panel(q);
        const int t = tid - 128, c0 = q * S::SB;
        if (p.a_rs == 1 || p.a_rs == -1) {
#pragma unroll
            for (int u = 0; u < S::SB / 4; ++u) {
                const int l = (t >> 5) + 4 * u;
                const double* src = A + (c0 + l) * p.a_cs + (c0 + lane) * p.a_rs;
                for (int i = c0 + lane; i < bs; i += 32, src += 32 * p.a_rs)
                    if (i > c0 + l) cp_async8(dst + l * S::LDT + i, src);
            }
        } else {
            const int l = t & 15;
            const double* src = A + (c0 + l) * p.a_cs + (c0 + (t >> 4)) * p.a_rs;
#pragma unroll 4
            for (int i = c0 + (t >> 4); i < bs; i += 8, src += 8 * p.a_rs)
                if (i > c0 + l) cp_async8(dst + l * S::LDT + i, src);
        }
    };
    if (warp >= 4) load(0);
    const bool c_row_fast = p.c_rs == 1 || p.c_rs == -1;
#pragma unroll
    for (int u = 0; u < C; ++u) {
        const int e = tid + u * S::NT;
        const int i = c_row_fast ? e % S::B : e / C, c = c_row_fast ? e / S::B : e % C;
        sC[i * C + c] = i < bs && c < nc ? a.alpha * Cp[i * p.c_rs + c * p.c_cs] : 0.0;
    }
    sD[tid] = tid < bs && !p.unit ? 1.0 / A[tid * (p.a_rs + p.a_cs)] : 1.0;
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();

    for (int q = 0; q < nq; ++q) {
        const int s0 = q * S::SB;
        if (warp == 0) {
            // (rows past the leaf: zeros, or stale words of M, in their own rows only)
            const int sc = lane / S::L, sg = lane % S::L;
            const double* m = panel(q) + s0 + sg;
            double x[S::RU];
#pragma unroll
            for (int u = 0; u < S::RU; ++u) x[u] = sC[(s0 + sg + S::L * u) * C + sc];
#pragma unroll
            for (int j = 0; j < S::SB; ++j) {
                const double xj =
                    __shfl_sync(0xffffffffu, x[j / S::L], j % S::L, S::L) * sD[s0 + j];
                if (sg == j % S::L) x[j / S::L] = xj;
#pragma unroll
                for (int u = j / S::L; u < S::RU; ++u)
                    if (sg + S::L * u > j) x[u] = fma(-m[j * S::LDT + S::L * u], xj, x[u]);
            }
#pragma unroll
            for (int u = 0; u < S::RU; ++u) sC[(s0 + sg + S::L * u) * C + sc] = x[u];
        } else if (warp < 4) {
            // block q - 1's columns off the rows from block q + 1 on
            const int n = q > 0 ? (bs - s0 - S::SB) * C : 0;
            const double* m = panel(q + S::STAGES - 1) + s0 + S::SB;
            const double* x = sC + (s0 - S::SB) * C;
            double* y = sC + (s0 + S::SB) * C;
            for (int o = tid - 32; o < n; o += 192) {
                const bool two = o + 96 < n;
                const int o1 = two ? o + 96 : o;
                double y0 = 0.0, y1 = 0.0;
#pragma unroll
                for (int kk = 0; kk < S::SB; ++kk) {
                    const double xv = x[kk * C + o % C];
                    y0 = fma(-m[kk * S::LDT + o / C], xv, y0);
                    if (two) y1 = fma(-m[kk * S::LDT + o1 / C], xv, y1);
                }
                // (16 products before they meet the row: its roundings stay as few as
                // with an update between smaller leaves)
                y[o] += y0;
                if (two) y[o1] += y1;
            }
        } else if (q + 1 < nq) {
            load(q + 1);
            asm volatile("cp.async.wait_all;" ::: "memory");
        }
        __syncthreads();
        if (q + 1 == nq) break;
        if (warp < 4) {
            // block q's columns off block q + 1
            const int kg = tid % S::KS, o = tid / S::KS;
            const double* m = panel(q) + s0 + S::SB + o / C;
            double* y = sC + (s0 + S::SB) * C + o;
            double acc = 0.0;
#pragma unroll
            for (int kk = 0; kk < S::SB; kk += S::KS)
                acc = fma(-m[(kk + kg) * S::LDT], sC[(s0 + kk + kg) * C + o % C], acc);
#pragma unroll
            for (int w = 1; w < S::KS; w *= 2) acc += __shfl_xor_sync(0xffffffffu, acc, w);
            if (kg == 0) *y += acc;
            asm volatile("bar.sync 1, 128;" ::: "memory");
        }
    }
#pragma unroll
    for (int u = 0; u < C; ++u) {
        const int e = tid + u * S::NT;
        const int i = c_row_fast ? e % S::B : e / C, c = c_row_fast ? e / S::B : e % C;
        if (i < bs && c < nc) Cp[i * p.c_rs + c * p.c_cs] = sC[i * C + c];
    }
}

}  // namespace

cudaError_t leaf64_configure() {
    cudaError_t e;
    if ((e = cudaFuncSetAttribute(leaf64_kernel<8>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)Leaf64<8>::smem)) != cudaSuccess)
        return e;
    return cudaFuncSetAttribute(leaf64_kernel<16>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)Leaf64<16>::smem);
}

cudaError_t leaf256_configure() {
    cudaError_t e;
    if ((e = cudaFuncSetAttribute(leaf256_kernel<2>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)Leaf256<2>::smem)) != cudaSuccess ||
        (e = cudaFuncSetAttribute(leaf256_kernel<4>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)Leaf256<4>::smem)) != cudaSuccess)
        return e;
    return cudaFuncSetAttribute(leaf256_kernel<8>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)Leaf256<8>::smem);
}

template <int C>
static cudaError_t leaf256_launch_c(const LeafArgs<double>& a, cudaStream_t s) {
    return launch_kernel(leaf256_kernel<C>, dim3((unsigned)((a.p.nrhs + C - 1) / C)),
                         dim3(Leaf256<C>::NT), Leaf256<C>::smem, s, a);
}
// Columns a CTA so that there is about one CTA an SM: each brings in all of M.
cudaError_t leaf256_launch(const LeafArgs<double>& a, int num_sms, cudaStream_t s) {
    if (a.p.nrhs <= 2 * (int64_t)num_sms) return leaf256_launch_c<2>(a, s);
    if (a.p.nrhs <= 4 * (int64_t)num_sms) return leaf256_launch_c<4>(a, s);
    return leaf256_launch_c<8>(a, s);
}

cudaError_t leaf64_launch(const LeafArgs<double>& a, int num_sms, cudaStream_t s) {
    const int c = a.p.nrhs <= 8 * (int64_t)num_sms ? 8 : 16;
    const dim3 grid((unsigned)((a.p.nrhs + c - 1) / c));
    if (c == 8) return launch_kernel(leaf64_kernel<8>, grid, dim3(128), Leaf64<8>::smem, s, a);
    return launch_kernel(leaf64_kernel<16>, grid, dim3(128), Leaf64<16>::smem, s, a);
}

}  // namespace trx
