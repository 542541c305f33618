// Problem descriptor of the batched kernels (canonical form, api.cu makes them).
#pragma once
#include <stdint.h>

namespace trx {

struct BatchDesc {
    int64_t k, nrhs;
    const void* A;
    int64_t a_rs, a_cs;
    void* C;
    int64_t c_rs, c_cs;
    double alpha;
    int unit, trsm, sb;        // trsm: 1 TRSM, 0 TRMM, 2 C := 0; sb: FP64 block height
    int bucket : 16;           // host: its problem's tuning bucket,
    int problems : 16;         // and 1 on a problem's first descriptor
};

constexpr int kBatchOrder = 512;   // largest order

constexpr int kBatchF64Chunk = 16;   // right-hand sides of the FP64 kernel's chunk
// Right-hand sides of the FP32 kernel's widest chunk at order k.
__host__ __device__ constexpr int64_t batch_f32_chunk(int64_t k) { return k <= 256 ? 64 : 32; }

}  // namespace trx
