// State-update kernels on FP32 SIMT cores.
//
//  * k_plain_1q / k_plain_2q: one launch per gate (the "plain FP32 per-gate"
//    baseline). Each thread moves 128-bit vectors: for a target above qubit 0,
//    two neighbouring pairs (quads) share one float4 per operand row; for a
//    target at qubit 0 the pair itself is one float4. HBM-bound: 16 * 2^n bytes
//    per gate against 8 (1q) or 16 (2q) real flop per amplitude, i.e. 0.5 or 1
//    flop per byte, far below the FP32 ridge.
//  * k_fused_simt<K>: one launch per fused K-qubit unitary (K <= 4). Thread =
//    one slice of 2^K amplitudes (the amplitudes that differ only in the target
//    bits); lanes of a warp take consecutive slices, so each copy covers
//    consecutive addresses along the lowest qubits. The unitary travels in the
//    kernel's parameter space (constant bank) and the fully unrolled complex
//    mat-vec reads it as constant operands. 8 * 2^K real flop per amplitude:
//    HBM-bound up to K = 4 on GB300 (at K = 4 just so: the packed multiply-adds
//    reach 68 TFLOP/s with nothing else to do, 253 us of a pass of 340).
//  * k_fused_wide<K>: fused K = 5, 6 or 7 qubit unitaries, a CTA per tile of 128,
//    64 or 32 slices, U from a device image in shared memory (see below).
//    Bound by the FP32 FMA pipe.
#include <algorithm>

#include "dev_common.cuh"
#include "internal.h"

namespace rcs {

struct Mat2 {
    float2 m[4];
};
struct Mat4 {
    float2 m[16];
};

constexpr int kUnroll = 4;

template <bool T0>
__global__ void __launch_bounds__(256) k_plain_1q(float2 *__restrict__ psi, uint64_t items, int t, Mat2 M) {
    const uint64_t stride = uint64_t(gridDim.x) * blockDim.x;
    const uint64_t hstep = 1ull << t;
    for (uint64_t it0 = uint64_t(blockIdx.x) * blockDim.x + threadIdx.x; it0 < items; it0 += stride * kUnroll) {
        float4 lo[kUnroll], hi[kUnroll];
        uint64_t idx[kUnroll];
#pragma unroll
        for (int u = 0; u < kUnroll; ++u) {
            const uint64_t it = it0 + u * stride;
            if (it < items) {
                if (T0) {
                    idx[u] = it * 2;
                    lo[u] = *reinterpret_cast<const float4 *>(psi + idx[u]);
                } else {
                    idx[u] = insert_zero(it * 2, t);
                    lo[u] = *reinterpret_cast<const float4 *>(psi + idx[u]);
                    hi[u] = *reinterpret_cast<const float4 *>(psi + idx[u] + hstep);
                }
            }
        }
#pragma unroll
        for (int u = 0; u < kUnroll; ++u) {
            const uint64_t it = it0 + u * stride;
            if (it >= items) continue;
            if (T0) {
                float2 a0 = make_float2(lo[u].x, lo[u].y), a1 = make_float2(lo[u].z, lo[u].w);
                float2 b0 = cmac(cmac(make_float2(0.f, 0.f), M.m[0], a0), M.m[1], a1);
                float2 b1 = cmac(cmac(make_float2(0.f, 0.f), M.m[2], a0), M.m[3], a1);
                *reinterpret_cast<float4 *>(psi + idx[u]) = make_float4(b0.x, b0.y, b1.x, b1.y);
            } else {
                float2 a0 = make_float2(lo[u].x, lo[u].y), a1 = make_float2(hi[u].x, hi[u].y);
                float2 c0 = make_float2(lo[u].z, lo[u].w), c1 = make_float2(hi[u].z, hi[u].w);
                float2 b0 = cmac(cmac(make_float2(0.f, 0.f), M.m[0], a0), M.m[1], a1);
                float2 b1 = cmac(cmac(make_float2(0.f, 0.f), M.m[2], a0), M.m[3], a1);
                float2 d0 = cmac(cmac(make_float2(0.f, 0.f), M.m[0], c0), M.m[1], c1);
                float2 d1 = cmac(cmac(make_float2(0.f, 0.f), M.m[2], c0), M.m[3], c1);
                *reinterpret_cast<float4 *>(psi + idx[u]) = make_float4(b0.x, b0.y, d0.x, d0.y);
                *reinterpret_cast<float4 *>(psi + idx[u] + hstep) = make_float4(b1.x, b1.y, d1.x, d1.y);
            }
        }
    }
}

__device__ __forceinline__ void mv4(const Mat4 &M, const float2 a[4], float2 b[4]) {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        float2 s = make_float2(0.f, 0.f);
#pragma unroll
        for (int l = 0; l < 4; ++l) s = cmac(s, M.m[j * 4 + l], a[l]);
        b[j] = s;
    }
}

// Two-qubit gate on qubits lo < hi, local index j = bit(lo) + 2 bit(hi).
template <bool LO0>
__global__ void __launch_bounds__(256) k_plain_2q(float2 *__restrict__ psi, uint64_t items, int lo, int hi,
                                                   Mat4 M) {
    const uint64_t stride = uint64_t(gridDim.x) * blockDim.x;
    const uint64_t sl = 1ull << lo, sh = 1ull << hi;
    for (uint64_t it0 = uint64_t(blockIdx.x) * blockDim.x + threadIdx.x; it0 < items; it0 += stride * 2) {
        float4 v[2][4];
        uint64_t base[2];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const uint64_t it = it0 + u * stride;
            if (it >= items) continue;
            if (LO0) {
                base[u] = insert_zero(insert_zero(it, 0), hi);
                v[u][0] = *reinterpret_cast<const float4 *>(psi + base[u]);       // j = 0, 1
                v[u][1] = *reinterpret_cast<const float4 *>(psi + base[u] + sh);  // j = 2, 3
            } else {
                base[u] = insert_zero(insert_zero(it * 2, lo), hi);
                v[u][0] = *reinterpret_cast<const float4 *>(psi + base[u]);
                v[u][1] = *reinterpret_cast<const float4 *>(psi + base[u] + sl);
                v[u][2] = *reinterpret_cast<const float4 *>(psi + base[u] + sh);
                v[u][3] = *reinterpret_cast<const float4 *>(psi + base[u] + sl + sh);
            }
        }
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const uint64_t it = it0 + u * stride;
            if (it >= items) continue;
            if (LO0) {
                float2 a[4] = {make_float2(v[u][0].x, v[u][0].y), make_float2(v[u][0].z, v[u][0].w),
                               make_float2(v[u][1].x, v[u][1].y), make_float2(v[u][1].z, v[u][1].w)};
                float2 b[4];
                mv4(M, a, b);
                *reinterpret_cast<float4 *>(psi + base[u]) = make_float4(b[0].x, b[0].y, b[1].x, b[1].y);
                *reinterpret_cast<float4 *>(psi + base[u] + sh) = make_float4(b[2].x, b[2].y, b[3].x, b[3].y);
            } else {
                // float4 e holds quads q (x,y) and q+1 (z,w) of operand row e
                float2 a[4], c[4], b[4], d[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    a[e] = make_float2(v[u][e].x, v[u][e].y);
                    c[e] = make_float2(v[u][e].z, v[u][e].w);
                }
                mv4(M, a, b);
                mv4(M, c, d);
                const uint64_t off[4] = {0, sl, sh, sl + sh};
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    *reinterpret_cast<float4 *>(psi + base[u] + off[e]) = make_float4(b[e].x, b[e].y, d[e].x, d[e].y);
            }
        }
    }
}

// Complex matrix entry as the two packed operands of its multiply-adds, precomputed on
// the host: rr = (re, re) and ni = (-im, im). With (x, y) an input amplitude, the packed
// FP32x2 fused multiply-adds acc += rr * (x, y) and acc += ni * (y, x) form
// (acc.x + re x - im y, acc.y + re y + im x): per component the same two fused
// multiply-adds, in the same order, as four scalar ones, in half the instructions.
struct CEnt {
    float2 rr, ni;
};

// Slice-order addressing, in bytes: a unit's base | a lane's base | a local amplitude's
// offset. The offsets and U are constant operands.
template <int K>
struct SimtArgs {
    CEnt U[1 << K][1 << K];
    uint64_t joff[1 << K];        // local amplitude j
    uint64_t coff[1 << (K - 1)];  // copy c of a unit (see k_fused_simt)
    uint64_t units;
    uint32_t depth;               // units in a warp's ring, 2..kSimtSlots
    uint32_t step;                // width 4: the CTA's warps start each unit together
    uint32_t flip;                // XORed into the unit numbers: 0, or units - 1 to walk the state backwards
    int t[K];                     // ascending
    int8_t rpos[5];               // index bit of lane (slice) bit i: the 5 lowest non-target qubits
    int8_t upos[32];              // index bit of unit number bit i: the other qubits (-1: none)
};

// CTAs of 8 warps per SM. At width 1 a unit is 512 bytes, and two CTAs do not keep enough in
// flight (371 against 326 us at 27 qubits); at width 4 three slow HBM down (340 against 370).
template <int K>
constexpr int simt_blocks_per_sm() {
    return K == 1 ? 3 : 2;
}
template <int K>
constexpr uint32_t simt_unit_bytes() {
    return 256u << K;  // 32 slices of 2^K amplitudes
}
constexpr uint32_t kSimtSlots = 3;  // of a warp's ring
// Units a warp keeps in its ring: the one it multiplies and one or two in flight. HBM serves
// wide copies best with no more in flight than it needs. At 27 qubits, two against three:
// width 4 with the lowest target on bits 1..4 340 and 350 us, with none below bit 5 360 and 335;
// width 3 330 and 360; width 2 360 and 326 (one 8-byte copy per amplitude through L1, one slice
// per thread in flight: 351-361, 342-347, 330-335).
template <int K>
uint32_t simt_depth(int lowest) {
    return K == 3 || (K == 4 && lowest < 5) ? 2u : 3u;
}
// Whether the warps of a CTA start each unit together at width 4, where multiplying a unit takes
// a warp nearly as long as HBM takes to serve it. Left alone they drift apart, and in a large
// state the copies of neighbouring units no longer come together: ms a pass at 32 qubits, alone
// and in step, targets on the top bits 11.9-12.1 and 11.2, in the middle 11.6-11.7 and 10.7,
// spread from bit 0 up 11.6 and 10.8 (one slice per thread, 8-byte copies: 11.4, 11.0, 11.2); at
// 28 qubits 698-710 and 678 us, 669-715 and 678, 708 and 664. At 27 the first two take 340 and
// 343, 333 and 342 us (the third 354 and 335), and at 25 and 26 they are slower in step as well.
// With the lowest target on bits 1 to 4 it costs 4 to 6% from 24 qubits on, and with targets on
// bits 0 and 1 together 15 to 25%.
bool simt_in_step(int n, int lowest, bool quad) { return n >= 28 && (lowest >= 5 || (lowest == 0 && !quad)); }

// A warp applies U to a unit of 32 neighbouring slices, one per lane, persistent over the
// units (grid-stride). Units come through a ring of shared-memory slots of the warp's own, so
// the copies of the next ones are in flight while it multiplies, and no block barrier is
// needed (simt_in_step says where there is one all the same). Copies are 16 bytes wide and bypass L1: for each pair of amplitudes (j = 2 c,
// 2 c + 1, which differ in the lowest target) the unit's 64 values are one 512-byte block in
// the order of their index bits: bit tb is the lowest target (bit 5 if that lies above bit 4),
// the others are the lane bits. So the lanes of a copy go up both in memory and in the slot.
// With tb = 2 or 3 the blocks' lines 1 and 3 have their halves or sectors swapped, which keeps
// the reads on different banks; with targets on bits 0 and 1 (quad) neighbouring lanes take
// the two halves of a 32-byte sector, amplitudes 4 i .. 4 i + 3 of one slice. Outputs leave in
// 16 bytes (32 in quad) while the lowest target is below bit 5: a slice's j, j + 1 where that
// is bit 0, else lane pairs swap one output and store two slices' j (even lane) or j + 1.
template <int K>
__global__ void __launch_bounds__(256, simt_blocks_per_sm<K>())
    k_fused_simt(float2 *__restrict__ psi, const __grid_constant__ SimtArgs<K> a) {
    constexpr int D = 1 << K;
    constexpr uint32_t kUnit = simt_unit_bytes<K>();
    extern __shared__ __align__(16) unsigned char simt_smem[];
    grid_trigger();
    const int lane = threadIdx.x & 31;
    const uint32_t warps = gridDim.x * 8u;
    const int tb = a.t[0] < 5 ? a.t[0] : 5;
    const bool quad = K > 1 && a.t[0] == 0 && a.t[K > 1] == 1;
    const bool odd = lane & 1;
    auto row = [&](int r) {
        uint64_t o = 0;
#pragma unroll
        for (int i = 0; i < 5; ++i)
            if ((r >> i) & 1) o |= 8ull << a.rpos[i];
        return o;
    };
    // copies: this lane's first value of a block, and its place in the slot
    const uint32_t swl = (tb == 2 || tb == 3) ? ((uint32_t(lane) >> 3) & 1u) << (tb - 1) : 0u;
    const int cs0 = quad ? lane >> 1 : ((2 * lane) & ((1 << tb) - 1)) | (((2 * lane) >> (tb + 1)) << tb);
    const uint64_t cbase =
        row(cs0) | (quad ? (odd ? a.joff[K > 1 ? 2 : 0] : 0ull) : (((2 * lane) >> tb) & 1) ? a.joff[1] : 0ull);
    unsigned char *ring = simt_smem + (threadIdx.x >> 5) * (kSimtSlots * kUnit);
    const uint32_t cdst = uint32_t(__cvta_generic_to_shared(ring)) + ((uint32_t(lane) ^ swl) << 4);
    // reads: where this lane's slice sits in a block, j even and j odd (quad: j mod 4 < 2 and >= 2)
    uint32_t rd0 = ((uint32_t(lane) >> tb) << (tb + 1)) | (uint32_t(lane) & ((1u << tb) - 1u));
    if (tb == 2 || tb == 3) rd0 ^= ((rd0 >> 4) & 1u) << tb;
    rd0 *= 8u;
    uint32_t rd1 = rd0 ^ (8u << tb);
    if (quad) {
        rd0 = (uint32_t(lane) & 15u) * 32u + (uint32_t(lane) >> 4) * 512u;
        rd1 = rd0 + 16u;
    }
    // stores
    const int smode = quad ? 3 : tb == 0 ? 1 : tb < 5 ? 2 : 0;
    const uint64_t sbase = row(smode == 2 ? lane & ~1 : lane) | (smode == 2 && odd ? a.joff[1] : 0ull);
    const int up = a.upos[lane];
    const uint64_t ubit = up >= 0 ? 8ull << up : 0ull;
    auto unit_base = [&](uint32_t u) {
        const bool on = ((u ^ a.flip) >> lane) & 1u;
        const uint32_t lo = __reduce_or_sync(0xffffffffu, on ? uint32_t(ubit) : 0u);
        const uint32_t hi = __reduce_or_sync(0xffffffffu, on ? uint32_t(ubit >> 32) : 0u);
        return (uint64_t(hi) << 32) | lo;
    };
    auto issue = [&](uint32_t u, uint32_t slot) {
        if (u < a.units) {
            const unsigned char *p = reinterpret_cast<const unsigned char *>(psi) + (cbase | unit_base(u));
#pragma unroll
            for (int c = 0; c < D / 2; ++c)
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(cdst + slot * kUnit + uint32_t(c) * 512u),
                             "l"(p + a.coff[c])
                             : "memory");
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    auto st16 = [](unsigned char *p, float2 x, float2 y) {
        asm volatile("st.global.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(p), "f"(x.x), "f"(x.y), "f"(y.x), "f"(y.y)
                     : "memory");
    };
    const uint32_t first = blockIdx.x * 8u;
    uint32_t u = first + (threadIdx.x >> 5);
    const bool deep = a.depth == 3;
    const bool step = K == 4 && a.step;
    grid_wait();  // the pass before (launch_after)
    issue(u, 0);
    if (deep) issue(u + warps, 1);
    uint32_t slot = 0, fill = deep ? 2 : 1;
#pragma unroll 1
    for (uint32_t c = first; c < a.units; c += warps, u += warps) {  // as many trips for every warp of the CTA
        if (step) __syncthreads();
        else __syncwarp();  // every lane has read the slot that is filled next
        if (u >= a.units) continue;  // fewer than 8 units
        issue(u + (deep ? 2 : 1) * warps, fill);
        if (++fill == a.depth) fill = 0;
        if (deep) asm volatile("cp.async.wait_group 2;" ::: "memory");  // this unit's copies
        else asm volatile("cp.async.wait_group 1;" ::: "memory");
        __syncwarp();  // ... and the other lanes'
        const unsigned char *in = ring + slot * kUnit;
        if (++slot == a.depth) slot = 0;
        float2 v[D], w[D];  // each input and its swapped form (y, x)
        if (tb == 0) {
#pragma unroll
            for (int j = 0; j < D; j += 2) {
                const float4 x = *reinterpret_cast<const float4 *>(
                    in + (quad ? ((j & 2) ? rd1 : rd0) + uint32_t(j / 4) * 1024u : rd0 + uint32_t(j / 2) * 512u));
                v[j] = make_float2(x.x, x.y);
                v[j + 1] = make_float2(x.z, x.w);
            }
        } else {
#pragma unroll
            for (int j = 0; j < D; ++j)
                v[j] = *reinterpret_cast<const float2 *>(in + ((j & 1) ? rd1 : rd0) + uint32_t(j / 2) * 512u);
        }
#pragma unroll
        for (int j = 0; j < D; ++j) w[j] = make_float2(v[j].y, v[j].x);
        unsigned char *out = reinterpret_cast<unsigned char *>(psi) + (sbase | unit_base(u));
        float2 held[4];  // outputs j & ~3 .. j
#pragma unroll
        for (int j = 0; j < D; ++j) {
            float2 acc = make_float2(0.f, 0.f);
#pragma unroll
            for (int l = 0; l < D; ++l) {
                const CEnt &e = a.U[j][l];
                acc = __ffma2_rn(e.rr, v[l], acc);
                acc = __ffma2_rn(e.ni, w[l], acc);
            }
            held[j & 3] = acc;
            if (smode == 0) {
                *reinterpret_cast<float2 *>(out + a.joff[j]) = acc;
            } else if (j & 1) {
                const float2 x = held[(j & 3) - 1], y = held[j & 3];
                if (smode == 1) {
                    st16(out + a.joff[j - 1], x, y);
                } else if (smode == 2) {
                    const float2 send = odd ? x : y;
                    const float2 recv = make_float2(__shfl_xor_sync(0xffffffffu, send.x, 1),
                                                    __shfl_xor_sync(0xffffffffu, send.y, 1));
                    st16(out + a.joff[j - 1], odd ? recv : x, odd ? y : recv);
                } else if ((j & 3) == 3) {
                    asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(out + a.joff[j & ~3]),
                                 "f"(held[0].x), "f"(held[0].y), "f"(held[1].x), "f"(held[1].y), "f"(held[2].x),
                                 "f"(held[2].y), "f"(held[3].x), "f"(held[3].y)
                                 : "memory");
                }
            }
        }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
}

// States of fewer than 32 slices (n < K + 5): one slice per thread, straight from memory.
template <int K>
__global__ void k_fused_small(float2 *__restrict__ psi, uint64_t slices, const __grid_constant__ SimtArgs<K> a) {
    constexpr int D = 1 << K;
    const uint64_t s = uint64_t(blockIdx.x) * blockDim.x + threadIdx.x;
    grid_trigger();
    grid_wait();
    if (s >= slices) return;
    uint64_t b = s;
#pragma unroll
    for (int i = 0; i < K; ++i) b = insert_zero(b, a.t[i]);
    float2 v[D], w[D];
#pragma unroll
    for (int j = 0; j < D; ++j) {
        v[j] = psi[b + a.joff[j] / 8];
        w[j] = make_float2(v[j].y, v[j].x);
    }
#pragma unroll
    for (int j = 0; j < D; ++j) {
        float2 acc = make_float2(0.f, 0.f);
#pragma unroll
        for (int l = 0; l < D; ++l) {
            acc = __ffma2_rn(a.U[j][l].rr, v[l], acc);
            acc = __ffma2_rn(a.U[j][l].ni, w[l], acc);
        }
        psi[b + a.joff[j] / 8] = acc;
    }
}

// ---- k_fused_wide<K>: fused 5- to 7-qubit unitaries on FP32 SIMT cores.
//
// From K = 5 a 2^K x 2^K complex matrix no longer fits the constant cache (as packed
// operands it is 16 KB at K = 5), and from K = 6 not the parameter space or a thread's
// registers, so a CTA applies it to a tile of T consecutive slices as a small complex
// GEMM in shared memory: out[s][j] = sum_l U[j][l] in[s][l], FP32 fused multiply-adds
// over l in increasing order. U comes from a device image laid out [l][j] (float2 re, im) and
// is copied into shared memory once per CTA. 8 * 2^K real flop per amplitude (16 to 64
// flop/B): past the FP32 ridge, so these passes are bound by the FMA pipe.
//
// A warp computes RJ outputs of 32 RS slices, a lane its slices (lane + 32 r): the matrix
// entries are the same for all lanes, the inputs are neighbouring words, and the outputs go
// straight to memory in runs of 32 slices. Outputs are packed by twos: the image holds (re_j,
// re_j+1, im_j, im_j+1), one 16-byte broadcast read, and four packed FP32x2 multiply-adds with
// (x, x), (-y, -y), (y, y), (x, x) do both outputs' complex multiply-add, per component the same
// operations in the same order as scalar ones. Two tile buffers let the next tile's copies run
// under the whole of the current tile's multiply-adds, with one barrier per tile. (Before: 4 x 4
// and 4 x 8 outputs per thread across lanes, scalar, outputs regrouped through shared memory
// with three more barriers, and no second buffer at K = 7.) Measured at 27 qubits, before and
// after, us a pass: K = 5 851-911 and 739-757, K = 6 1371-1419 and 1306-1342, K = 7 2757-2787 and
// 2450-2484 (46, 53 and 56 TFLOP/s now; packed multiply-adds with nothing else to do reach 68).
constexpr int kWideThreads = 256;

// Per width: RS slices per lane, RJ outputs per warp; the warps of a group share slices, and
// the groups of a CTA split a tile's. Resident CTAs per SM, by shared memory: three at K = 5
// (72 KB), two at K = 6 (96 KB), one at K = 7 (192 KB).
template <int K>
struct WideShape {
    static constexpr int D = 1 << K;
    static constexpr int RS = K == 5 ? 2 : 1;
    static constexpr int RJ = K == 5 ? 8 : 16;
    static constexpr int Group = D / RJ;                         // warps of a group
    static constexpr int T = 32 * RS * (kWideThreads / 32 / Group);  // slices of a tile
    static constexpr int Blocks = K == 5 ? 3 : (K == 6 ? 2 : 1);
    static constexpr size_t Smem = size_t(D) * D * 8 + 2 * size_t(D) * T * 8 + size_t(D) * 8;
};

template <int K>
constexpr int wide_blocks_per_sm() {
    return WideShape<K>::Blocks;
}

template <int K>
constexpr size_t wide_smem_bytes() {
    return WideShape<K>::Smem;
}

struct WideArgs {
    int t[8];  // ascending targets (K used)
    uint64_t slices;
};

template <int K>
__global__ void __launch_bounds__(kWideThreads, wide_blocks_per_sm<K>())
    k_fused_wide(float2 *__restrict__ psi, const float2 *__restrict__ ut, const __grid_constant__ WideArgs a) {
    using S = WideShape<K>;
    constexpr int D = S::D, RS = S::RS, RJ = S::RJ, T = S::T;
    extern __shared__ __align__(16) unsigned char wide_smem[];
    float2 *U = reinterpret_cast<float2 *>(wide_smem);  // [l][j], packed by two outputs (simt_build_ops)
    float2 *buf = U + D * D;                             // two of [j][T]
    uint64_t *offs = reinterpret_cast<uint64_t *>(buf + 2 * D * T);
    const int tid = threadIdx.x;
    const uint64_t slices = a.slices;
    grid_trigger();
    for (int j = tid; j < D; j += kWideThreads) {
        uint64_t o = 0;
#pragma unroll
        for (int i = 0; i < K; ++i)
            if ((j >> i) & 1) o |= 1ull << a.t[i];
        offs[j] = o;
    }
    {  // U image: D * D * 8 bytes in 16-byte copies
        const uint32_t dst0 = uint32_t(__cvta_generic_to_shared(U));
        for (int c = tid; c < D * D / 2; c += kWideThreads)
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst0 + uint32_t(c) * 16u), "l"(ut + 2 * c)
                         : "memory");
        asm volatile("cp.async.commit_group;" ::: "memory");
    }
    __syncthreads();  // offs
    grid_wait();      // the pass before (launch_after); U came from the host
    const uint64_t ntiles = (slices + T - 1) / T;
    // copy walk: slice s = tid % T, rows j = tid / T + (256 / T) i
    const int ws = tid % T, wj = tid / T;
    // compute: slices s0 + 32 r, outputs j0 .. j0 + RJ - 1
    const int s0 = (tid & 31) + (tid >> 5) / S::Group * (32 * RS), j0 = (tid >> 5) % S::Group * RJ;
    const uint32_t buf0 = uint32_t(__cvta_generic_to_shared(buf));
    auto base_of = [&](uint64_t sl) {
        uint64_t b = sl;
#pragma unroll
        for (int i = 0; i < K; ++i) b = insert_zero(b, a.t[i]);
        return b;
    };
    auto issue = [&](uint64_t tile, int which) {
        const uint64_t sl = tile * T + uint64_t(ws);
        if (tile < ntiles && sl < slices) {
            const uint64_t b = base_of(sl);
            const uint32_t dst0 = buf0 + uint32_t(which * D * T) * 8u;
#pragma unroll 4
            for (int j = wj; j < D; j += kWideThreads / T) {
                const uint32_t dst = dst0 + uint32_t(j * T + ws) * 8u;
                asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(dst), "l"(psi + (b | offs[j])) : "memory");
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    int cur = 0;
    issue(blockIdx.x, 0);
#pragma unroll 1
    for (uint64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x, cur ^= 1) {
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncthreads();  // the tile has landed, and every thread is done with the other buffer
        issue(tile + gridDim.x, cur ^ 1);
        const float2 *bt = buf + cur * D * T + s0;
        const float4 *u4 = reinterpret_cast<const float4 *>(U + j0);
        float2 X[RS][RJ / 2], Y[RS][RJ / 2];  // real and imaginary parts of outputs j, j + 1
#pragma unroll
        for (int r = 0; r < RS; ++r)
#pragma unroll
            for (int c = 0; c < RJ / 2; ++c) X[r][c] = Y[r][c] = make_float2(0.f, 0.f);
#pragma unroll 2
        for (int l = 0; l < D; ++l) {
            float2 x[RS];
            float4 u[RJ / 2];
#pragma unroll
            for (int r = 0; r < RS; ++r) x[r] = bt[l * T + 32 * r];
#pragma unroll
            for (int c = 0; c < RJ / 2; ++c) u[c] = u4[l * (D / 2) + c];
#pragma unroll
            for (int r = 0; r < RS; ++r) {
                const float2 xx = make_float2(x[r].x, x[r].x), yy = make_float2(x[r].y, x[r].y),
                             ny = make_float2(-x[r].y, -x[r].y);
#pragma unroll
                for (int c = 0; c < RJ / 2; ++c) {
                    const float2 re = make_float2(u[c].x, u[c].y), im = make_float2(u[c].z, u[c].w);
                    X[r][c] = __ffma2_rn(re, xx, X[r][c]);
                    X[r][c] = __ffma2_rn(im, ny, X[r][c]);
                    Y[r][c] = __ffma2_rn(re, yy, Y[r][c]);
                    Y[r][c] = __ffma2_rn(im, xx, Y[r][c]);
                }
            }
        }
#pragma unroll
        for (int r = 0; r < RS; ++r) {
            const uint64_t s = tile * T + uint64_t(s0 + 32 * r);
            if (s < slices) {
                float2 *p = psi + base_of(s);
#pragma unroll
                for (int c = 0; c < RJ / 2; ++c) {
                    p[offs[j0 + 2 * c]] = make_float2(X[r][c].x, Y[r][c].x);
                    p[offs[j0 + 2 * c + 1]] = make_float2(X[r][c].y, Y[r][c].y);
                }
            }
        }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
}

__global__ void k_init_zero(float4 *__restrict__ psi4, uint64_t n4) {
    grid_trigger();
    grid_wait();
    const uint64_t stride = uint64_t(gridDim.x) * blockDim.x;
    for (uint64_t i = uint64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < n4; i += stride)
        psi4[i] = make_float4(i == 0 ? 1.f : 0.f, 0.f, 0.f, 0.f);
}

static int check_launch() { return launch_status("state-update kernel"); }

// Full state from a compact sub-state: psi[i] = sub[c(i)] when every bit of i outside
// tmask is 0 (c(i) gathers the bits of i at the positions of tmask, in order), else 0.
// A circuit started from |0...0> leaves every qubit its first passes do not touch in
// |0>, so those passes can run on the 2^popcount(tmask) sub-state and this one write
// pass replaces the reset and them. c(i) is assembled from the runs of consecutive
// bits of tmask: run r moves the bits (i & mask[r]) down by shift[r] to its place in
// c, so a few shifts replace a loop over every bit of tmask (which made the kernel
// issue-bound: 22 ms from a 30- to a 32-qubit sub-state, 1.8 TB/s).
constexpr int kExpandRuns = 32;  // a 64-bit mask holds at most 32 runs of ones
struct ExpandArgs {
    uint64_t tmask;
    uint64_t mask[kExpandRuns];
    int runs;
    uint8_t shift[kExpandRuns];
};

// One thread per output float4 (amplitudes 2f and 2f + 1). With bit 0 in tmask both
// come from sub[c], sub[c + 1] (c even: one 16-byte load); without it 2f + 1 is 0.
__global__ void k_expand(float4 *__restrict__ psi4, uint64_t n4, const float2 *__restrict__ sub,
                         const __grid_constant__ ExpandArgs a) {
    const uint64_t stride = uint64_t(gridDim.x) * blockDim.x;
    const bool pair = a.tmask & 1ull;
    grid_trigger();
    grid_wait();
    for (uint64_t f = uint64_t(blockIdx.x) * blockDim.x + threadIdx.x; f < n4; f += stride) {
        const uint64_t i0 = 2 * f;
        float4 out = make_float4(0.f, 0.f, 0.f, 0.f);
        if (!(i0 & ~a.tmask)) {
            uint64_t c = 0;
            for (int r = 0; r < a.runs; ++r) c |= (i0 & a.mask[r]) >> a.shift[r];
            if (pair) {
                out = __ldg(reinterpret_cast<const float4 *>(sub) + (c >> 1));
            } else {
                const float2 v = __ldg(sub + c);
                out = make_float4(v.x, v.y, 0.f, 0.f);
            }
        }
        psi4[f] = out;
    }
}

int launch_expand(void *psi, int n, const void *sub, uint64_t tmask, void *stream) {
    if (n < 1 || (reinterpret_cast<uintptr_t>(sub) & 15u))
        return note_launch_refusal(RCS_ERR_ARG, "state expansion: bad size or a sub-state not 16-byte aligned");
    ExpandArgs a{};
    a.tmask = tmask;
    int placed = 0;  // bits of tmask below the current run
    for (int q = 0; q < 64;) {
        if (!((tmask >> q) & 1)) {
            ++q;
            continue;
        }
        int len = 0;
        while (q + len < 64 && ((tmask >> (q + len)) & 1)) ++len;
        a.mask[a.runs] = (len == 64 ? ~0ull : ((1ull << len) - 1ull)) << q;
        a.shift[a.runs] = uint8_t(q - placed);
        ++a.runs;
        placed += len;
        q += len;
    }
    const uint64_t n4 = (1ull << n) / 2;
    const cudaError_t e = launch_after(k_expand, grid_for(n4, 256, device_sm_count(), 8), 256, 0,
                                       static_cast<cudaStream_t>(stream), static_cast<float4 *>(psi), n4,
                                       static_cast<const float2 *>(sub), a);
    return e == cudaSuccess ? RCS_OK : note_launch_error("state expansion", e);
}

int launch_init_zero(void *psi, int n, void *stream) {
    auto st = static_cast<cudaStream_t>(stream);
    if (n == 0) return RCS_ERR_ARG;
    const uint64_t n4 = (1ull << n) / 2;  // n >= 1: whole float4s
    const cudaError_t e =
        launch_after(k_init_zero, grid_for(n4, 256, device_sm_count(), 8), 256, 0, st, static_cast<float4 *>(psi), n4);
    return e == cudaSuccess ? RCS_OK : note_launch_error("zero state", e);
}

int launch_pass_plain(void *psi, int n, const Pass &p, void *stream) {
    auto st = static_cast<cudaStream_t>(stream);
    auto *s = static_cast<float2 *>(psi);
    const int sms = device_sm_count();
    if (p.kind == PASS_1Q) {
        Mat2 M;
        for (int e = 0; e < 4; ++e) M.m[e] = make_float2(float(p.U[e].real()), float(p.U[e].imag()));
        const int t = p.t[0];
        if (t == 0) {
            const uint64_t items = 1ull << (n - 1);
            k_plain_1q<true><<<grid_for(items, 256, sms, 8), 256, 0, st>>>(s, items, t, M);
        } else {
            const uint64_t items = 1ull << (n - 2);
            k_plain_1q<false><<<grid_for(items, 256, sms, 8), 256, 0, st>>>(s, items, t, M);
        }
    } else if (p.kind == PASS_2Q) {
        Mat4 M;
        for (int e = 0; e < 16; ++e) M.m[e] = make_float2(float(p.U[e].real()), float(p.U[e].imag()));
        const int lo = p.t[0], hi = p.t[1];
        if (lo == 0) {
            const uint64_t items = 1ull << (n - 2);
            k_plain_2q<true><<<grid_for(items, 256, sms, 8), 256, 0, st>>>(s, items, lo, hi, M);
        } else {
            const uint64_t items = 1ull << (n - 3);
            k_plain_2q<false><<<grid_for(items, 256, sms, 8), 256, 0, st>>>(s, items, lo, hi, M);
        }
    } else {
        return RCS_ERR_ARG;
    }
    return check_launch();
}

// Dynamic shared memory of a fused pass's launch whose kernel needs `smem`: so much that no SM
// takes more than its even share of the CTAs. They come in (launch_after) while those of the
// passes before sit on most SMs; without this they crowded onto the others, as many to an SM as
// fit, and the pass took as much longer. Back to back on 19 qubits, us a pass: width 5 (128
// CTAs) 9.6 to 20.2 (by its targets), now 5.7 to 9.9; width 6 (128) 13.5 to 20.2, now 8.5 to
// 12.1; width 3 (256) 4.5 to 4.8, now 3.6 to 3.7. On 20 qubits width 5 (256) 11.8 to 24.6, now
// 8.9 to 16.5. Without overlap with the pass before: 8.5 to 12.7, 10.7 to 14.7, 6.4, 10.7 to 18.8.
constexpr size_t kSmemPerSm = 228 * 1024;  // each CTA takes 1 KB of it for the system
static size_t spread_smem(size_t smem, unsigned grid) {
    const unsigned sms = unsigned(device_sm_count()), share = (grid + sms - 1) / sms;
    return std::max(smem, kSmemPerSm / (share + 1));
}

// Shared-memory attribute of k_fused_simt<K> on the current device (once).
template <int K>
static int simt_attr() {
    static bool attr_done[64] = {};
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev >= 0 && dev < 64 && attr_done[dev]) return RCS_OK;
    const cudaError_t e = cudaFuncSetAttribute(k_fused_simt<K>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                               int(std::max(kSmemPerSm / 2, size_t(8 * kSimtSlots * simt_unit_bytes<K>()))));
    if (e != cudaSuccess) return note_launch_error("fused kernel shared-memory attribute", e);
    if (dev >= 0 && dev < 64) attr_done[dev] = true;
    return RCS_OK;
}

// Shared-memory attribute of k_fused_wide<K> on the current device (once).
template <int K>
static int wide_attr() {
    static bool attr_done[64] = {};
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev >= 0 && dev < 64 && attr_done[dev]) return RCS_OK;
    const cudaError_t e =
        cudaFuncSetAttribute(k_fused_wide<K>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             int(std::max(kSmemPerSm / 2, wide_smem_bytes<K>())));
    if (e != cudaSuccess) return note_launch_error("wide fused kernel shared-memory attribute", e);
    if (dev >= 0 && dev < 64) attr_done[dev] = true;
    return RCS_OK;
}

int simt_prepare_device() {
    int rc = simt_attr<1>();
    if (rc == RCS_OK) rc = simt_attr<2>();
    if (rc == RCS_OK) rc = simt_attr<3>();
    if (rc == RCS_OK) rc = simt_attr<4>();
    if (rc == RCS_OK) rc = wide_attr<5>();
    if (rc == RCS_OK) rc = wide_attr<6>();
    if (rc == RCS_OK) rc = wide_attr<7>();
    return rc;
}

size_t simt_ops_bytes(int k) { return k > kSimtParamK ? size_t(8) << (2 * k) : 0; }

// FP32 image of a wide pass, l-major: per l and pair of outputs j, j + 1 (j even) the real
// parts of U[j][l] and U[j + 1][l], then their imaginary parts.
void simt_build_ops(const Pass &p, uint8_t *out) {
    const int D = 1 << p.k;
    auto *f = reinterpret_cast<float *>(out);
    for (int l = 0; l < D; ++l)
        for (int j = 0; j < D; ++j) {
            const cd &u = p.U[size_t(j) * D + l];
            float *at = f + 2 * (size_t(l) * D + (j & ~1)) + (j & 1);
            at[0] = float(u.real());
            at[2] = float(u.imag());
        }
}

template <int K>
static int launch_simt_k(float2 *psi, int n, const Pass &p, bool backwards, cudaStream_t st) {
    SimtArgs<K> a;
    const int D = 1 << K;
    for (int i = 0; i < K; ++i) a.t[i] = p.t[i];
    for (int j = 0; j < D; ++j) {
        a.joff[j] = 0;
        for (int i = 0; i < K; ++i)
            if ((j >> i) & 1) a.joff[j] |= 8ull << p.t[i];
        for (int l = 0; l < D; ++l) {
            const cd &u = p.U[size_t(j) * D + l];
            a.U[j][l] = CEnt{make_float2(float(u.real()), float(u.real())), make_float2(-float(u.imag()), float(u.imag()))};
        }
    }
    if (n < K + 5) {
        const uint64_t slices = 1ull << (n - K);
        const cudaError_t e = launch_after(k_fused_small<K>, 1, 32, 0, st, psi, slices, a);
        return e == cudaSuccess ? RCS_OK : note_launch_error("fused pass", e);
    }
    std::fill(a.upos, a.upos + 32, int8_t(-1));
    for (int qb = 0, i = 0; qb < n; ++qb) {
        if (std::find(p.t, p.t + K, qb) != p.t + K) continue;
        if (i < 5) a.rpos[i] = int8_t(qb);
        else a.upos[i - 5] = int8_t(qb);
        ++i;
    }
    const bool quad = K > 1 && p.t[0] == 0 && p.t[1] == 1;
    for (int c = 0; c < D / 2; ++c)
        a.coff[c] = quad ? ((c & 1) ? 8ull << a.rpos[4] : 0ull) + a.joff[4 * (c >> 1)] : a.joff[2 * c];
    a.units = 1ull << (n - K - 5);
    a.flip = backwards ? uint32_t(a.units - 1) : 0u;
    a.step = K == 4 && simt_in_step(n, p.t[0], quad);
    a.depth = a.step ? 2u : simt_depth<K>(p.t[0]);
    if (int rc = simt_attr<K>(); rc != RCS_OK) return rc;
    // persistent: the resident CTAs, never more than the units need
    const unsigned grid = grid_for(a.units, 8, device_sm_count(), simt_blocks_per_sm<K>());
    const size_t smem = spread_smem(8 * kSimtSlots * simt_unit_bytes<K>(), grid);
    const cudaError_t e = launch_after(k_fused_simt<K>, grid, 256, smem, st, psi, a);
    return e == cudaSuccess ? RCS_OK : note_launch_error("fused pass", e);
}

template <int K>
static int launch_wide_k(float2 *psi, int n, const Pass &p, const uint8_t *ops, cudaStream_t st) {
    if (!ops || (reinterpret_cast<uintptr_t>(ops) & 15u))
        return note_launch_refusal(RCS_ERR_ARG, "fused pass of width 5..7 without a 16-byte aligned U image");
    WideArgs a{};
    for (int i = 0; i < K; ++i) a.t[i] = p.t[i];
    a.slices = 1ull << (n - K);
    if (int rc = wide_attr<K>(); rc != RCS_OK) return rc;
    const uint64_t tiles = (a.slices + WideShape<K>::T - 1) / WideShape<K>::T;
    const uint64_t resident = uint64_t(device_sm_count()) * wide_blocks_per_sm<K>();
    const unsigned grid = unsigned(tiles < resident ? tiles : resident);
    const size_t smem = spread_smem(wide_smem_bytes<K>(), grid);
    const cudaError_t e = launch_after(k_fused_wide<K>, grid, kWideThreads, smem, st, psi,
                                       reinterpret_cast<const float2 *>(ops), a);
    return e == cudaSuccess ? RCS_OK : note_launch_error("wide fused pass", e);
}

int launch_pass_simt(void *psi, int n, const Pass &p, const uint8_t *ops, void *stream, bool backwards) {
    auto st = static_cast<cudaStream_t>(stream);
    auto *s = static_cast<float2 *>(psi);
    if (p.k > n) return RCS_ERR_ARG;
    switch (p.k) {
        case 1: return launch_simt_k<1>(s, n, p, backwards, st);
        case 2: return launch_simt_k<2>(s, n, p, backwards, st);
        case 3: return launch_simt_k<3>(s, n, p, backwards, st);
        case 4: return launch_simt_k<4>(s, n, p, backwards, st);
        case 5: return launch_wide_k<5>(s, n, p, ops, st);
        case 6: return launch_wide_k<6>(s, n, p, ops, st);
        case 7: return launch_wide_k<7>(s, n, p, ops, st);
        default: return RCS_ERR_UNSUPPORTED;
    }
}

}  // namespace rcs
