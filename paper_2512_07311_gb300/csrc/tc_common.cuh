// Shapes, shared-memory layout constants and MMA wrappers shared by the tensor-core
// kernels that apply one 64 x 64 unitary per pass (the single-pass kernel and the
// persistent batch kernel): M = 128 slices per tile, K = N = 128 reals, the BF16
// realified and TF32 complex-block operand images, and the instruction descriptors.
#pragma once

#include <cstdint>

#include "dev_common.cuh"
#include "internal.h"
#include "tc_ptx.cuh"

namespace rcs {

namespace tc {
constexpr int K = kTcK;         // 6 target qubits
constexpr int D = 1 << K;       // 64 amplitudes per slice
constexpr int KR = 2 * D;       // 128 reals per slice (GEMM K)
constexpr int NR = 2 * D;       // 128 real outputs (GEMM N)
constexpr int M = 128;          // slices per tile (GEMM M, TMEM lanes)
constexpr int kLoaderWarps = 8;
constexpr int kEpiWarps = 8;
constexpr int kThreads = (kLoaderWarps + kEpiWarps + 1) * 32;  // 544
// Chains of passes (k_tc.cu).
constexpr int kChainMax = 3;                    // passes of a chain
constexpr int kChainThreads = kThreads + 64;    // two more warps order the chunks
// From 128 MB a state no longer stays in L2 from one pass to the next (two passes at 24 qubits:
// 87 us as a chain, 95 one after the other; at 23 qubits 57 against 47).
constexpr int kChainMinQubits = 24;
// Amplitudes of a chunk: 8 MB, 128 tiles, one to three for each CTA of a pass. Every two passes fit
// one (their targets and seven lowest other qubits are at most 19), three do where they share
// enough. The larger a chunk, the fewer of them fit the window below. Measured with chunks of at
// least 2^18 / 2^19 / 2^20 / 2^21: the 30-qubit, 14-cycle circuit 35.6 / 32.9 / 32.1 / 32.9 ms,
// the 27-qubit, 20-cycle one 5.72 / 5.23 / 5.19 / 5.31.
constexpr int kChunkLog2 = 20;
// Distance between two passes of a chain. The tiles in flight in both (about 4 per SM each) and
// the counters' round trip take some 70 MB; beyond about 80 MB for a pair and 64 MB a step for
// three the chunks start to fall out of L2. Measured at 27 qubits, us a pass: pairs with 40 /
// 56 / 72 / 80 / 96 / 128 MB 301 / 259 / 233 / 229 / 248 / 288; threes with 20 / 32 / 48 / 64 MB
// 416 / 289 / 243 / 230.
constexpr uint64_t kChainWindowBytes[kChainMax + 1] = {0, 0, uint64_t(80) << 20, uint64_t(64) << 20};
// Time of a chain in passes of one launch each, for splitting a sequence: pairs and threes take
// about 0.7 a pass (229 to 238 against 323 us at 27 qubits), a pass left over a whole one.
constexpr double kChainCost[kChainMax + 1] = {0, 1.0, 1.36, 2.06};
constexpr int kOpBytes = NR * KR * 2;                          // one bf16 operand image: 32 KB
constexpr int kStageBytes = D * M * 8;                         // one tile of complex64: 64 KB
constexpr int kSmBhi = 0;                                      // BF16: B_hi image, then B_lo
constexpr int kSmBlo = kOpBytes;
// TF32: per split (hi, lo) one K-major image of the 192 x 64 matrix [-Ui; Ur; Ui]
// (rows = outputs, K = inputs), in two 128-byte swizzle atom columns of 32 inputs.
constexpr int kTf32Rows = 3 * D;
constexpr int kTf32Atom = kTf32Rows * 128;   // 24 KB
constexpr int kTf32Split = 2 * kTf32Atom;    // 48 KB
constexpr int kSlotBytes = 4096;  // slice-order loaders: one unit of 16 amplitudes x 32 slices
// Shared-memory map (offsets from a 1024-aligned base): the B images, the stage (two of
// one tile each, or kSlots units per loader warp), then the small tables.
template <bool kTf32>
struct Layout {
    static constexpr int kBBytes = kTf32 ? 2 * kTf32Split : 2 * kOpBytes;
    static constexpr int kStage0 = kBBytes;
    static constexpr int kSlots = kTf32 ? 4 : 5;  // what fits beside the B images
    static constexpr int kOff = kStage0 + kLoaderWarps * kSlots * kSlotBytes;  // 64 x u64 target offsets
    static constexpr int kHiOff = kOff + D * 8;             // 64 x u64 offsets of the high compact bits
    static constexpr int kCj = kHiOff + 64 * 8;             // 64 x u16 compact index of local amplitude j
    static constexpr int kCs = kCj + D * 2;                 // 128 x u16 compact index of slice s within the tile
    static constexpr int kBar = kCs + M * 2;                // 16 mbarriers
    static constexpr int kMisc = kBar + 16 * 8;             // tmem slot, abort flag, chain: chunk limit, 8 counts
    static constexpr int kAlloc = kMisc + 48 + 1024;        // slack for 1024-byte alignment
    static_assert(kAlloc <= 227 * 1024, "shared memory");
    static_assert(kLoaderWarps * kSlots * kSlotBytes >= 2 * kStageBytes, "the stage of the other variants");
};
constexpr uint32_t kTmemCols = 512;
// instruction descriptor: D f32, A bf16, B bf16, both K-major, N = 128, M = 128
constexpr uint32_t kIdesc = (1u << 4) | (1u << 7) | (1u << 10) | (uint32_t(NR >> 3) << 17) | (uint32_t(M >> 4) << 24);
// TF32 variant: D f32, A tf32, B tf32, both K-major, N = 128 (Re outputs, then Im), M = 128
constexpr uint32_t kIdescTf32 = (1u << 4) | (2u << 7) | (2u << 10) | (uint32_t(128 >> 3) << 17) | (uint32_t(M >> 4) << 24);
}  // namespace tc

__device__ __forceinline__ void mma_bf16_tmemA(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t accum) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}" ::"r"(d_tmem),
        "r"(a_tmem), "l"(b_desc), "r"(tc::kIdesc), "r"(accum)
        : "memory");
}

__device__ __forceinline__ void mma_tf32_tmemA(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc,
                                               uint32_t accum) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::tf32 [%0], [%1], %2, %3, p;\n\t}" ::"r"(d_tmem),
        "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accum)
        : "memory");
}

__device__ __forceinline__ uint64_t slice_base(uint64_t s, const int (&t)[tc::K]) {
#pragma unroll
    for (int i = 0; i < tc::K; ++i) s = insert_zero(s, t[i]);
    return s;
}

}  // namespace rcs
