// Changes of the stored qubit layout: an in-place permutation of the index bits of a
// state, and the copy of a caller-order range out of a permuted one.
//
// k_permute: psi[x] <- psi[m(x)], where m moves index bits. A tile is the set of
// amplitudes that differ only in the bits B = (bit 0, the moved bits and the lowest others,
// 12 in all): m maps each tile to itself, so a CTA reads a tile into shared memory, and
// writes it back in the new order: one read and one write of the state however many bits
// move. Bit 0 is in B, so global loads and stores are 16 bytes wide. The layouts that the
// planner chooses swap up to 5 low bits with high ones, so bits 1..4 are in B too and runs
// are at least 2^5 amplitudes; a loaded file may move 11 high bits in a pass, whose runs are
// then 2 amplitudes, half a sector. The shared index is XOR-swizzled (its bits 4..7 and
// 8..11 folded onto bits 0..3), which keeps reads along bits that differ mod 4 on different
// banks. Measured (a planned layout, 3 swaps): 8.1 us at 19 qubits, 555 us at 27,
// where one trip through HBM takes 321: the eight float4 that a thread holds do not fit the
// 40 registers of six CTAs per SM, and spill (DRAM 2.7 GB instead of 2.1; shared-memory
// pipe 51% busy). The exchange of circuit qubits with the lowest bits used to run as one
// k_plain_2q pass per swap: 1.35 ms for 4 swaps at 27 qubits.
#include <algorithm>
#include <bit>

#include "dev_common.cuh"
#include "internal.h"

namespace rcs {

constexpr int kPermBits = 12;     // log2 of the tile: 32 KB
constexpr int kPermThreads = 256;  // 8 index bits of float4s; the tile's other 3 are walked
constexpr int kPermIters = (1 << kPermBits) / 2 / kPermThreads;

struct PermArgs {
    float4 *psi;
    uint64_t tiles;
    uint32_t f4;                // float4s of a tile (fewer than 2^11 below 12 qubits)
    int8_t tpos[32];            // index bit of tile number bit i, or -1
    int8_t bpos[kPermBits];     // index bit of tile-local bit i (ascending; bpos[0] = 0)
    uint16_t from[kPermBits];   // swizzled shared index of the old place of new local bit i
    uint64_t ioff[kPermIters];  // float4 offset of walk step i
    uint16_t isrc[kPermIters];  // ... and its swizzled old place
};

__host__ __device__ inline uint32_t perm_swizzle(uint32_t x) { return x ^ ((x >> 4) & 15u) ^ ((x >> 8) & 15u); }

__global__ void __launch_bounds__(kPermThreads, 6) k_permute(const __grid_constant__ PermArgs a) {
    __shared__ float2 tile[1 << kPermBits];
    const int lane = threadIdx.x & 31;
    // this thread's float4 is local index 2 tid (+ 512 per walk step)
    uint64_t off = 0;
    uint32_t src = 0;
#pragma unroll
    for (int i = 0; i < 8; ++i)
        if ((threadIdx.x >> i) & 1) {
            off |= 1ull << (a.bpos[i + 1] - 1);
            src ^= a.from[i + 1];
        }
    const int tp = a.tpos[lane];
    const uint64_t tbit = tp >= 0 ? 1ull << (tp - 1) : 0ull;  // in float4s
    for (uint64_t t = blockIdx.x; t < a.tiles; t += gridDim.x) {
        const bool on = (t >> lane) & 1ull;
        const uint32_t lo = __reduce_or_sync(0xffffffffu, on ? uint32_t(tbit) : 0u);
        const uint32_t hi = __reduce_or_sync(0xffffffffu, on ? uint32_t(tbit >> 32) : 0u);
        float4 *p = a.psi + (off | (uint64_t(hi) << 32) | lo);
        float4 v[kPermIters];
#pragma unroll
        for (int i = 0; i < kPermIters; ++i)
            if (threadIdx.x + i * kPermThreads < a.f4) v[i] = p[a.ioff[i]];
#pragma unroll
        for (int i = 0; i < kPermIters; ++i)
            if (threadIdx.x + i * kPermThreads < a.f4) {
                const uint32_t x = perm_swizzle(2u * (threadIdx.x + i * kPermThreads));
                tile[x] = make_float2(v[i].x, v[i].y);
                tile[x ^ 1u] = make_float2(v[i].z, v[i].w);
            }
        __syncthreads();
#pragma unroll
        for (int i = 0; i < kPermIters; ++i)
            if (threadIdx.x + i * kPermThreads < a.f4) {
                const uint32_t x = src ^ a.isrc[i];
                const float2 y = tile[x], z = tile[x ^ a.from[0]];
                p[a.ioff[i]] = make_float4(y.x, y.y, z.x, z.y);
            }
        __syncthreads();  // the next tile overwrites the buffer
    }
}

// One permutation pass: new index bit b comes from old index bit m[b]. The moved bits and
// bit 0 must fit a tile.
static int launch_permute(void *psi, int n, const int *m, cudaStream_t st) {
    uint64_t B = 1;
    for (int b = 0; b < n; ++b)
        if (m[b] != b) B |= 1ull << b;
    const int nb = std::min(n, kPermBits);
    for (int b = 0; b < n && std::popcount(B) < nb; ++b) B |= 1ull << b;
    if (n < 1 || std::popcount(B) > kPermBits) return note_launch_refusal(RCS_ERR_ARG, "layout permutation too wide");
    PermArgs a{};
    a.psi = static_cast<float4 *>(psi);
    a.tiles = 1ull << (n - nb);
    a.f4 = (1u << nb) / 2;
    int local[64];
    std::fill(a.tpos, a.tpos + 32, int8_t(-1));
    std::fill(a.bpos, a.bpos + kPermBits, int8_t(1));  // unused bits: never set in a live thread
    int nt = 0, nl = 0;
    for (int b = 0; b < n; ++b) {
        if ((B >> b) & 1) {
            local[b] = nl;
            a.bpos[nl++] = int8_t(b);
        } else {
            a.tpos[nt++] = int8_t(b);
        }
    }
    for (int i = 0; i < nb; ++i) a.from[i] = uint16_t(perm_swizzle(1u << local[m[a.bpos[i]]]));
    for (int i = 0; i < kPermIters; ++i)
        for (int k = 0; k < 3; ++k)
            if (((i >> k) & 1) && 9 + k < nb) {
                a.ioff[i] |= 1ull << (a.bpos[9 + k] - 1);
                a.isrc[i] = uint16_t(a.isrc[i] ^ a.from[9 + k]);
            }
    const unsigned grid = unsigned(std::min<uint64_t>(a.tiles, uint64_t(device_sm_count()) * 6));
    k_permute<<<grid, kPermThreads, 0, st>>>(a);
    return launch_status("layout permutation");
}

int launch_restore_layout(void *psi, int n, int *phys_of, void *stream) {
    int phys[64], log_of[64], m[64];
    for (int q = 0; q < n; ++q) {
        phys[q] = phys_of[q];
        log_of[phys[q]] = q;
        m[q] = q;
    }
    // swaps of two index bits that bring every qubit home, gathered into passes of up to a
    // tile's bits (a planned layout needs one pass; a longer permutation several)
    uint64_t moved = 1;
    auto flush = [&]() {
        int rc = RCS_OK;
        if (moved != 1) rc = launch_permute(psi, n, m, static_cast<cudaStream_t>(stream));
        if (rc == RCS_OK) std::copy(phys, phys + n, phys_of);
        for (int q = 0; q < n; ++q) m[q] = q;
        moved = 1;
        return rc;
    };
    for (int p = 0; p < n; ++p)
        while (log_of[p] != p) {
            const int l = log_of[p], q = phys[p];  // qubit p sits at q, bit p holds qubit l
            const uint64_t both = (1ull << p) | (1ull << q);
            if (std::popcount(moved | both) > kPermBits)
                if (int rc = flush(); rc != RCS_OK) return rc;
            moved |= both;
            std::swap(m[p], m[q]);
            phys[p] = p;
            phys[l] = q;
            log_of[p] = p;
            log_of[q] = l;
        }
    return flush();
}

// out[i] = psi[map(first + i)]: a range in the caller's order, one thread per amplitude.
__global__ void __launch_bounds__(256) k_read_mapped(const float2 *__restrict__ psi, uint64_t first, uint64_t count,
                                                     const BitMap map, float2 *__restrict__ out) {
    const uint64_t stride = uint64_t(gridDim.x) * blockDim.x;
    for (uint64_t i = uint64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < count; i += stride)
        out[i] = __ldg(psi + map_bits(map, first + i));
}

int launch_read_mapped(const void *psi, uint64_t first, uint64_t count, const BitMap &map, void *out, void *stream) {
    if (count == 0) return RCS_OK;
    k_read_mapped<<<grid_for(count, 256, device_sm_count(), 8), 256, 0, static_cast<cudaStream_t>(stream)>>>(
        static_cast<const float2 *>(psi), first, count, map, static_cast<float2 *>(out));
    return launch_status("mapped read");
}

}  // namespace rcs
