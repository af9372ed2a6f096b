// Expert construction: RTN quantizer, packer, canonical import / export.
//
// Section 3.1 of the paper: the experts are quantized variants of one
// full-precision model, built once and frozen.  The quantizer is affine
// round-to-nearest per (output channel, group of input features); see moqe.h
// for the exact arithmetic.  What decides a code, scale or zero-point is a single
// IEEE operation (explicit __f*_rn intrinsics, no fast math; see round_chunk),
// so they are reproducible bit for bit.
#include <cstdio>
#include <cstring>
#include <mutex>
#include <new>

#include "dequant.cuh"
#include "ptx.cuh"

namespace moqe {
namespace {

// ---------------------------------------------------------------------------
// piece <-> packed words
// ---------------------------------------------------------------------------
// code index i = 8*G + t  (chunk G, position t)  <->  k = 128*kb + 32*G + 8*q + t
template <int BITS>
__device__ __forceinline__ void encode_piece(const uint32_t (&c)[32], uint32_t (&w)[PieceWords<BITS>::n]) {
    if constexpr (BITS == 4) {
#pragma unroll
        for (int G = 0; G < 4; ++G) {
            uint32_t v = 0;
#pragma unroll
            for (int t = 0; t < 8; ++t) {
                int nib = (t & 1) ? 4 + (t >> 1) : (t >> 1);
                v |= (c[8 * G + t] & 0xFu) << (4 * nib);
            }
            w[G] = v;
        }
    } else if constexpr (BITS == 2) {
        w[0] = w[1] = 0;
#pragma unroll
        for (int i = 0; i < 32; ++i) {
            const int G = i >> 3, t = i & 7;
            w[G >> 1] |= (c[i] & 3u) << (2 * (4 * (G & 1) + (t >> 1)) + 16 * (t & 1));
        }
    } else if constexpr (BITS == 8) {
#pragma unroll
        for (int j = 0; j < 8; ++j)
            w[j] = (c[4 * j] & 0xFFu) | ((c[4 * j + 1] & 0xFFu) << 8) | ((c[4 * j + 2] & 0xFFu) << 16) |
                   ((c[4 * j + 3] & 0xFFu) << 24);
    } else {
        w[0] = w[1] = w[2] = 0;
#pragma unroll
        for (int i = 0; i < 30; ++i) {
            int p = i >> 1;
            w[p / 5] |= (c[i] & 7u) << (3 * (p % 5) + 16 * (i & 1));
        }
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            w[b] |= ((c[30] >> b) & 1u) << 15;
            w[b] |= ((c[31] >> b) & 1u) << 31;
        }
    }
}

template <int BITS>
__device__ __forceinline__ void decode_piece(const uint32_t (&w)[PieceWords<BITS>::n], uint32_t (&c)[32]) {
    if constexpr (BITS == 4) {
#pragma unroll
        for (int G = 0; G < 4; ++G)
#pragma unroll
            for (int t = 0; t < 8; ++t) {
                int nib = (t & 1) ? 4 + (t >> 1) : (t >> 1);
                c[8 * G + t] = (w[G] >> (4 * nib)) & 0xFu;
            }
    } else if constexpr (BITS == 2) {
#pragma unroll
        for (int i = 0; i < 32; ++i) {
            const int G = i >> 3, t = i & 7;
            c[i] = (w[G >> 1] >> (2 * (4 * (G & 1) + (t >> 1)) + 16 * (t & 1))) & 3u;
        }
    } else if constexpr (BITS == 8) {
#pragma unroll
        for (int i = 0; i < 32; ++i) c[i] = (w[i >> 2] >> (8 * (i & 3))) & 0xFFu;
    } else {
#pragma unroll
        for (int i = 0; i < 30; ++i) {
            int p = i >> 1;
            c[i] = (w[p / 5] >> (3 * (p % 5) + 16 * (i & 1))) & 7u;
        }
        c[30] = c[31] = 0;
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            c[30] |= ((w[b] >> 15) & 1u) << b;
            c[31] |= ((w[b] >> 31) & 1u) << b;
        }
    }
}

// address of the words of piece (half, slot) inside a blob
template <int BITS>
__device__ __forceinline__ void store_piece(uint8_t* blob, int half, int slot, const uint32_t (&w)[PieceWords<BITS>::n]) {
    if constexpr (BITS == 4) {
        *reinterpret_cast<uint4*>(blob + half * 512 + slot * 16) = make_uint4(w[0], w[1], w[2], w[3]);
    } else if constexpr (BITS == 2) {
        *reinterpret_cast<uint2*>(blob + slot * 16 + half * 8) = make_uint2(w[0], w[1]);
    } else if constexpr (BITS == 8) {
        *reinterpret_cast<uint4*>(blob + half * 1024 + slot * 16) = make_uint4(w[0], w[1], w[2], w[3]);
        *reinterpret_cast<uint4*>(blob + half * 1024 + 512 + slot * 16) = make_uint4(w[4], w[5], w[6], w[7]);
    } else {
        uint32_t* a = reinterpret_cast<uint32_t*>(blob + slot * 16);
        uint32_t* b = reinterpret_cast<uint32_t*>(blob + 512 + slot * 8);
        if (half == 0) { a[0] = w[0]; a[1] = w[1]; a[2] = w[2]; }
        else           { a[3] = w[0]; b[0] = w[1]; b[1] = w[2]; }
    }
}

template <int BITS>
__device__ __forceinline__ void load_piece(const uint8_t* blob, int half, int slot, uint32_t (&w)[PieceWords<BITS>::n]) {
    if constexpr (BITS == 4) {
        uint4 v = *reinterpret_cast<const uint4*>(blob + half * 512 + slot * 16);
        w[0] = v.x; w[1] = v.y; w[2] = v.z; w[3] = v.w;
    } else if constexpr (BITS == 2) {
        uint2 v = *reinterpret_cast<const uint2*>(blob + slot * 16 + half * 8);
        w[0] = v.x; w[1] = v.y;
    } else if constexpr (BITS == 8) {
        uint4 v = *reinterpret_cast<const uint4*>(blob + half * 1024 + slot * 16);
        uint4 u = *reinterpret_cast<const uint4*>(blob + half * 1024 + 512 + slot * 16);
        w[0] = v.x; w[1] = v.y; w[2] = v.z; w[3] = v.w; w[4] = u.x; w[5] = u.y; w[6] = u.z; w[7] = u.w;
    } else {
        const uint32_t* a = reinterpret_cast<const uint32_t*>(blob + slot * 16);
        const uint32_t* b = reinterpret_cast<const uint32_t*>(blob + 512 + slot * 8);
        if (half == 0) { w[0] = a[0]; w[1] = a[1]; w[2] = a[2]; }
        else           { w[0] = a[3]; w[1] = b[0]; w[2] = b[1]; }
    }
}

// piece id -> coordinates.  Pieces are numbered so that consecutive threads own
// consecutive slots of one half of one blob (coalesced packed accesses).
struct PieceCoord { int nt, kb, nb, half, slot, q, r, n; size_t tile_index; };
__device__ __forceinline__ PieceCoord piece_coord(long long pid, int KB) {
    PieceCoord pc;
    pc.slot = (int)(pid & 31);
    pc.half = (int)((pid >> 5) & 1);
    pc.nb = (int)((pid >> 6) & 7);
    long long tile = pid >> 9;
    pc.kb = (int)(tile % KB);
    pc.nt = (int)(tile / KB);
    pc.q = pc.slot >> 3;
    pc.r = (pc.slot & 7) ^ (2 * pc.q);
    pc.n = pc.nt * 128 + pc.nb * 16 + pc.half * 8 + pc.r;
    pc.tile_index = (size_t)tile;
    return pc;
}

// ---------------------------------------------------------------------------
// K1a: per (channel, group) scale and zero-point.  One warp per group.
// ---------------------------------------------------------------------------
// where the scale / zero-point of (channel n, canonical group gi) live; a group wider than 128 k is
// stored once per tile it spans: copy 0 .. copies-1
struct MetaSlot { __half* s; __nv_bfloat16* z; };
__device__ __forceinline__ int meta_copies(int group) { return group > 128 ? group / 128 : 1; }
__device__ __forceinline__ MetaSlot meta_slot(uint8_t* tiles, __half* scales_pc, __nv_bfloat16* zeros_pc, int bits, int group,
                                              int has_zeros, int KB, int n, int gi, int copy) {
    MetaSlot m;
    if (group == 0) {
        m.s = scales_pc + n;
        m.z = has_zeros ? zeros_pc + n : nullptr;
        return m;
    }
    const int per_tile = moqe_groups_per_tile(group);
    const int kb = group >= 128 ? gi * (group / 128) + copy : gi / per_tile;
    const int j = group >= 128 ? 0 : gi % per_tile;
    uint8_t* tile = tiles + ((size_t)(n >> 7) * KB + kb) * (size_t)moqe_tile_stride(bits, group, has_zeros);
    uint8_t* meta = tile + moqe_tile_bytes(bits) + j * moqe_meta_group_bytes(has_zeros);
    m.s = reinterpret_cast<__half*>(meta) + (n & 127);
    m.z = has_zeros ? reinterpret_cast<__nv_bfloat16*>(meta + 256) + (n & 127) : nullptr;
    return m;
}

// scale and zero-point of a group from its extremes, exactly as moqe.h states them
struct GroupGrid { __half sh; float s; int z; };
__device__ __forceinline__ GroupGrid group_grid(float lo, float hi, float a, int bits, int sym) {
    GroupGrid g;
    const int L = (1 << bits) - 1, qmax = (1 << (bits - 1)) - 1;
    const float s32 = sym ? __fdiv_rn(a, (float)qmax) : __fdiv_rn(__fsub_rn(hi, lo), (float)L);
    g.sh = __float2half_rn(s32);
    g.s = __half2float(g.sh);
    if (!(g.s > 0.f) || isinf(g.s)) { g.sh = __float2half_rn(1.0f); g.s = 1.0f; }
    g.z = sym ? 1 << (bits - 1) : max(0, min(L, (int)rintf(__fdiv_rn(-lo, g.s))));
    return g;
}

__global__ void rtn_scales_kernel(const float* __restrict__ W, int N, int K, int bits, int group, int G, int sym, int KB,
                                  uint8_t* __restrict__ tiles, __half* __restrict__ scales_pc,
                                  __nv_bfloat16* __restrict__ zeros_pc) {
    long long warp = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    int lane = threadIdx.x & 31;
    if (warp >= (long long)N * G) return;
    int n = (int)(warp / G), gi = (int)(warp % G);
    const int g = group ? group : K;
    const float* w = W + (size_t)n * K + (size_t)gi * g;
    float lo = 0.f, hi = 0.f, a = 0.f;
    for (int k = lane; k < g; k += 32) {
        float v = w[k];
        lo = fminf(lo, v);
        hi = fmaxf(hi, v);
        a = fmaxf(a, fabsf(v));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, o));
        hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, o));
        a = fmaxf(a, __shfl_xor_sync(0xffffffffu, a, o));
    }
    if (lane != 0) return;
    const GroupGrid g2 = group_grid(lo, hi, a, bits, sym);
    for (int c = 0; c < meta_copies(group); ++c) {
        MetaSlot m = meta_slot(tiles, scales_pc, zeros_pc, bits, group, !sym, KB, n, gi, c);
        *m.s = g2.sh;
        if (!sym) *m.z = __float2bfloat16_rn((float)g2.z);         // exact: z <= 255
    }
}

// ---------------------------------------------------------------------------
// K1b: codes + packing (FROM_CODES: canonical codes are given, only pack)
// ---------------------------------------------------------------------------
template <int BITS, bool FROM_CODES>
__global__ void encode_pack_kernel(const float* __restrict__ W, const uint8_t* __restrict__ canon, int N, int K,
                                   int g /*0 = per channel*/, int sym, int KB, uint8_t* __restrict__ tiles,
                                   __half* __restrict__ scales_pc, __nv_bfloat16* __restrict__ zeros_pc, long long npieces) {
    long long pid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (pid >= npieces) return;
    PieceCoord pc = piece_coord(pid, KB);
    constexpr int L = (1 << BITS) - 1;
    constexpr int half_code = 1 << (BITS - 1);
    constexpr int qmax = half_code - 1;
    uint32_t c[32];
#pragma unroll
    for (int G = 0; G < 4; ++G) {
        int k0 = pc.kb * 128 + 32 * G + 8 * pc.q;
        bool live = (pc.n < N) && (k0 < K);            // K % 8 == 0: a chunk is wholly inside or outside
        if (!live) {
#pragma unroll
            for (int t = 0; t < 8; ++t) c[8 * G + t] = 0;
            continue;
        }
        if constexpr (FROM_CODES) {
            uint2 v = *reinterpret_cast<const uint2*>(canon + (size_t)pc.n * K + k0);
#pragma unroll
            for (int t = 0; t < 4; ++t) {
                c[8 * G + t] = (v.x >> (8 * t)) & 0xFFu;
                c[8 * G + 4 + t] = (v.y >> (8 * t)) & 0xFFu;
            }
        } else {
            MetaSlot m = meta_slot(tiles, scales_pc, zeros_pc, BITS, g, !sym, KB, pc.n, g ? k0 / g : 0, 0);
            float s = __half2float(*m.s);
            int z = sym ? half_code : (int)__bfloat162float(*m.z);
            const float4* src = reinterpret_cast<const float4*>(W + (size_t)pc.n * K + k0);
            float4 v0 = src[0], v1 = src[1];
            float wv[8] = {v0.x, v0.y, v0.z, v0.w, v1.x, v1.y, v1.z, v1.w};
#pragma unroll
            for (int t = 0; t < 8; ++t) {
                int q = (int)rintf(__fdiv_rn(wv[t], s));   // (beyond an int where fp16 has no scale for the group: clamped before it is added to)
                if (sym) q = max(-qmax, min(qmax, q)) + half_code;
                else     q = max(0, min(L, min(L, q) + z));
                c[8 * G + t] = (uint32_t)q;
            }
        }
    }
    uint32_t w[PieceWords<BITS>::n];
    encode_piece<BITS>(c, w);
    store_piece<BITS>(tiles + pc.tile_index * (size_t)moqe_tile_stride(BITS, g, !sym) + pc.nb * moqe_blob_bytes(BITS), pc.half,
                      pc.slot, w);
}

// ---------------------------------------------------------------------------
// K1: scales, zero-points, codes and packing in one kernel: quantize_group_kernel for groups within a k-block,
// quantize_channel_kernel for per-channel experts (wider groups, and some of those, take K1a and K1b above, see one_kernel).
// Every byte of the tiles is written here, padding included.
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint64_t pack_f2(float lo, float hi) { uint64_t r; asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi)); return r; }
__device__ __forceinline__ float2 unpack_f2(uint64_t v) { float2 r; asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v)); return r; }
__device__ __forceinline__ uint64_t fma_f2(uint64_t a, uint64_t b, uint64_t c) { uint64_t r; asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c)); return r; }

// the nearest whole number, within 16 bits, so that a zero-point can be added to it (where fp16 has no scale for a group its scale is 1,
// and quotients may be beyond an int); 0 for NaN
__device__ __forceinline__ int rounded16(float x) { short q; asm("cvt.rni.s16.f32 %0, %1;" : "=h"(q) : "f"(x)); return q; }
// (the larger one, and NaN if either is)
__device__ __forceinline__ float max_or_nan(float a, float b) { float r; asm("max.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b)); return r; }

// what rounding a chunk of 8 weights needs of its group.  safe: no |w / s| of the group is large (see round_chunk)
struct Rounding { float s, inv; int z; bool safe; };
template <int BITS>
__device__ __forceinline__ Rounding rounding(const GroupGrid& g, float top) {
    const float inv = __frcp_rn(g.s);
    return {g.s, inv, g.z, top * inv < (float)(1 << (BITS + 1))};
}
// Codes of a chunk, in pairs of 16 bits: clamp(rint(w / s) + z) as IEEE division and rounding give rint(w / s), from a
// multiplication by 1 / s.  Adding 1.5 * 2^23 + z rounds w * inv to the nearest integer and leaves code and zero-point added up
// in the low bits: no conversion instructions, which run at a quarter of the rate.  The product is off by at most 2^-22 of its
// size; only where it comes that close to the middle between two integers (or is large, or no number) does the division decide.
template <int BITS>
__device__ __forceinline__ void round_chunk(const float* w, const Rounding& g, bool sym, uint32_t* pair) {
    constexpr int L = (1 << BITS) - 1, half_code = 1 << (BITS - 1);
    const float magic = 12582912.f + (float)g.z;                        // (a symmetric grid's z is half_code)
    const uint64_t inv2 = pack_f2(g.inv, g.inv), magic2 = pack_f2(magic, magic), minus = pack_f2(-1.f, -1.f);
    float worst = 0.f;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const uint64_t x = pack_f2(w[2 * j], w[2 * j + 1]), y = fma_f2(x, inv2, magic2);
        const float2 yy = unpack_f2(y), d = unpack_f2(fma_f2(x, inv2, fma_f2(y, minus, magic2)));     // d: the product less its integer
        worst = max_or_nan(worst, max_or_nan(fabsf(d.x), fabsf(d.y)));
        pair[j] = __byte_perm(__float_as_uint(yy.x), __float_as_uint(yy.y), 0x5410u);
    }
    if (!g.safe || !(worst < 0.5f - (float)(1 << (BITS + 1)) * 0x1p-21f)) {
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int a = rounded16(__fdiv_rn(w[2 * j], g.s)) + g.z, b = rounded16(__fdiv_rn(w[2 * j + 1], g.s)) + g.z;
            pair[j] = ((uint32_t)min(max(a, -1), L + 1) & 0xFFFFu) | (uint32_t)min(max(b, -1), L + 1) << 16;
        }
    }
    constexpr uint32_t L2 = (uint32_t)L * 0x10001u;
#pragma unroll
    for (int j = 0; j < 4; ++j) pair[j] = sym ? __vmins2(__vmaxs2(pair[j], 0x10001u), L2) : __vimin_s16x2_relu(pair[j], L2);
    static_assert(half_code >= 2, "a symmetric code is at least 1");
}
// the packed words of a piece from its codes in pairs (2 i, 2 i + 1): see encode_piece
template <int BITS>
__device__ __forceinline__ void encode_pairs(const uint32_t (&c)[16], uint32_t (&w)[PieceWords<BITS>::n]) {
    if constexpr (BITS == 8) {
#pragma unroll
        for (int j = 0; j < 8; ++j) w[j] = __byte_perm(c[2 * j], c[2 * j + 1], 0x6420u);
    } else if constexpr (BITS == 3) {
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            w[j] = c[5 * j];
#pragma unroll
            for (int f = 1; f < 5; ++f) w[j] |= c[5 * j + f] << (3 * f);
            w[j] |= (c[15] >> j & 0x10001u) << 15;
        }
    } else {
        constexpr int F = 16 / BITS;                                    // pairs to a word
#pragma unroll
        for (int j = 0; j < 16 / F; ++j) {
            w[j] = c[F * j];
#pragma unroll
            for (int f = 1; f < F; ++f) w[j] |= c[F * j + f] << (BITS * f);
        }
    }
}

// Groups of 32, 64 or 128 k.  Bound by the fp32 weights' bytes, read once.  A warp takes one blob, 16 channels x 128 k, after
// another, an unrelated one each time; the next two are on their way into its own two stages of shared memory (four boxes of 32
// k x 16 rows each: with the 128-byte swizzle a quarter-warp's eight rows fall on different banks), so that loads are always in
// flight and take no registers.  One block of 12 warps to an SM: 192 KB of stages.  11008 x 4096, 4-bit g128: 42 us, of which 28 are
// the weights' bytes at the copy rate; 57 with 24 warps an SM that load into registers and wait.  g32 74 (8 bit) and 70 (2 bit).
constexpr int QG_WARPS = 12, QG_STAGES = 2, QG_STAGE = 16 * 128 * 4;
constexpr int QG_SMEM = 1024 + QG_WARPS * QG_STAGES * QG_STAGE;
template <int BITS>
__global__ void __launch_bounds__(QG_WARPS * 32, 1) quantize_group_kernel(const __grid_constant__ CUtensorMap wmap, int N, int K, int group, int sym, int KB,
                                                                     long long blobs, uint8_t* __restrict__ tiles, int* status) {
    extern __shared__ unsigned char q_smem[];
    __shared__ unsigned long long bars[QG_WARPS * QG_STAGES];
    __shared__ int s_abort;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t smem0 = (smem_u32(q_smem) + 1023u & ~1023u) + warp * (QG_STAGES * QG_STAGE), bar0 = smem_u32(bars) + warp * QG_STAGES * 8;
    if (threadIdx.x == 0) s_abort = 0;
    if (lane == 0)
        for (int i = 0; i < QG_STAGES; ++i) mbar_init(bar0 + 8 * i, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    __syncthreads();
    const int q = lane >> 3, r = (lane & 7) ^ (2 * q);                  // this lane's slot: piece (q, r) of both halves
    const int stride = moqe_tile_stride(BITS, group, !sym), per = moqe_groups_per_tile(group), meta_g = moqe_meta_group_bytes(!sym);
    auto partner = [&](int d) { const int p = q ^ d; return p * 8 + (r ^ (2 * p)); };      // the lane that holds (q ^ d, r)
    const long long step = (long long)gridDim.x * QG_WARPS;
    auto fetch = [&](long long u, int stage) {                          // (by one lane)
        const long long strip = u / KB;
        const int k0 = (int)(u - strip * KB) * 128;
        mbar_expect_tx(bar0 + 8 * stage, QG_STAGE);
#pragma unroll
        for (int G = 0; G < 4; ++G)
            asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
                         ::"r"(smem0 + stage * QG_STAGE + G * (QG_STAGE / 4)), "l"(&wmap), "r"(k0 + 32 * G), "r"((int)strip * 16), "r"(bar0 + 8 * stage) : "memory");
    };
    const long long u0 = (long long)warp * gridDim.x + blockIdx.x;
    if (lane == 0)
        for (int i = 0; i < QG_STAGES; ++i)
            if (u0 + i * step < blobs) fetch(u0 + i * step, i);
    __syncwarp();
    int n = 0;
#pragma unroll 1
    for (long long u = u0; u < blobs; u += step, ++n) {
        const int stage = n % QG_STAGES;
        if (!__all_sync(0xffffffffu, mbar_wait_short(bar0 + 8 * stage, n / QG_STAGES & 1u, &s_abort, status))) break;
        const long long strip = u / KB;
        const int kb = (int)(u - strip * KB), nt = (int)(strip >> 3), nb = (int)(strip & 7);
        uint8_t* tile = tiles + ((size_t)nt * KB + kb) * (size_t)stride;
        const bool inside = nt * 128 + nb * 16 + 16 <= N && kb * 128 + 128 <= K;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int row = nt * 128 + nb * 16 + 8 * h + r;
            float v[32];                                                // (zeros outside of W)
#pragma unroll
            for (int G = 0; G < 4; ++G)
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    const uint32_t at = smem0 + stage * QG_STAGE + G * (QG_STAGE / 4) + (8 * h + r) * 128 + (((2 * q + i) ^ r) << 4);
                    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
                                 : "=f"(v[8 * G + 4 * i]), "=f"(v[8 * G + 4 * i + 1]), "=f"(v[8 * G + 4 * i + 2]), "=f"(v[8 * G + 4 * i + 3]) : "r"(at));
                }
            float lo[4], hi[4];
#pragma unroll
            for (int G = 0; G < 4; ++G) {
                lo[G] = hi[G] = 0.f;
#pragma unroll
                for (int t = 0; t < 8; ++t) { lo[G] = fminf(lo[G], v[8 * G + t]); hi[G] = fmaxf(hi[G], v[8 * G + t]); }
            }
            if (per < 4) {
                lo[0] = fminf(lo[0], lo[1]); hi[0] = fmaxf(hi[0], hi[1]);
                lo[2] = fminf(lo[2], lo[3]); hi[2] = fmaxf(hi[2], hi[3]);
            }
            if (per == 1) { lo[0] = fminf(lo[0], lo[2]); hi[0] = fmaxf(hi[0], hi[2]); }
            Rounding g[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                if (j < per) {
                    float l = lo[0], t = hi[0];
                    if (j > 0) {
                        l = per == 2 ? lo[2] : (j == 1 ? lo[1] : (j == 2 ? lo[2] : lo[3]));
                        t = per == 2 ? hi[2] : (j == 1 ? hi[1] : (j == 2 ? hi[2] : hi[3]));
                    }
#pragma unroll
                    for (int d = 1; d < 4; d <<= 1) {
                        l = fminf(l, __shfl_sync(0xffffffffu, l, partner(d)));
                        t = fmaxf(t, __shfl_sync(0xffffffffu, t, partner(d)));
                    }
                    const float top = fmaxf(-l, t);                     // (max |w|)
                    const GroupGrid gg = group_grid(l, t, top, BITS, sym);
                    const Rounding rr = rounding<BITS>(gg, top);
#pragma unroll
                    for (int G = 0; G < 4; ++G)
                        if (per == 1 || (per == 2 ? (G >> 1) == j : G == j)) g[G] = rr;
                    if (q == 0) {
                        const bool live = row < N && kb * 128 + j * (128 / per) < K;
                        uint8_t* m = tile + moqe_tile_bytes(BITS) + j * meta_g + (nb * 16 + 8 * h + r) * 2;
                        *reinterpret_cast<__half*>(m) = live ? gg.sh : __float2half_rn(0.f);
                        if (!sym) *reinterpret_cast<__nv_bfloat16*>(m + 256) = __float2bfloat16_rn(live ? (float)gg.z : 0.f);
                    }
                }
            }
            // (every lane has its values of the second half: its extremes went through the exchange above)
            if (h == 1 && lane == 0 && u + QG_STAGES * step < blobs) fetch(u + QG_STAGES * step, stage);
            uint32_t c[16], w[PieceWords<BITS>::n];
#pragma unroll
            for (int G = 0; G < 4; ++G) round_chunk<BITS>(v + 8 * G, g[G], sym, c + 4 * G);
            if (!inside) {
#pragma unroll
                for (int i = 0; i < 16; ++i)
                    if (row >= N || kb * 128 + 32 * (i >> 2) + 8 * q >= K) c[i] = 0u;      // K % 8 == 0: a chunk is wholly inside or outside
            }
            encode_pairs<BITS>(c, w);
            store_piece<BITS>(tile + nb * moqe_blob_bytes(BITS), h, lane, w);
        }
    }
    if (s_abort) {
        // let copies that may still be in flight land before the shared memory is released
        const unsigned long long t0 = global_ns();
        while (global_ns() - t0 < 200000ull) __nanosleep(1000);
    }
}

// Per channel.  A block goes over its 16 rows twice, the second time out of L2 (16 rows are 256 KB at K = 4096); a warp holds the
// 16 channels x 128 k of a blob in registers between loading and rounding.  BLOCKS: to an SM, see channel_blocks; with two a warp has
// both halves of a blob under way before it rounds the first.
template <int BITS, int BLOCKS>
__global__ void __launch_bounds__(256, BLOCKS) quantize_channel_kernel(const float* __restrict__ W, int N, int K, int sym, int KB,
                                                               uint8_t* __restrict__ tiles, __half* __restrict__ scales_pc,
                                                               __nv_bfloat16* __restrict__ zeros_pc) {
    __shared__ float s_ext[8][2][16];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int nt = blockIdx.x >> 3, nb = blockIdx.x & 7;
    const int q = lane >> 3, r = (lane & 7) ^ (2 * q);                  // this lane's slot: piece (q, r) of both halves
    const int row0 = nt * 128 + nb * 16 + r;
    const int stride = moqe_tile_stride(BITS, 0, !sym);
    // the lane that holds (q ^ d, r)
    auto partner = [&](int d) { const int p = q ^ d; return p * 8 + (r ^ (2 * p)); };
    auto load = [&](int n, int kb, float (&v)[32]) {
#pragma unroll
        for (int G = 0; G < 4; ++G) {
            const int k0 = kb * 128 + 32 * G + 8 * q;
            const bool live = n < N && k0 < K;                          // K % 8 == 0: a chunk is wholly inside or outside
            const float4* src = reinterpret_cast<const float4*>(W + (live ? (size_t)n * K + k0 : 0));
            const float4 a = live ? src[0] : make_float4(0.f, 0.f, 0.f, 0.f), b = live ? src[1] : make_float4(0.f, 0.f, 0.f, 0.f);
            v[8 * G] = a.x; v[8 * G + 1] = a.y; v[8 * G + 2] = a.z; v[8 * G + 3] = a.w;
            v[8 * G + 4] = b.x; v[8 * G + 5] = b.y; v[8 * G + 6] = b.z; v[8 * G + 7] = b.w;
        }
    };
    Rounding g[2];
    float lo[2] = {0.f, 0.f}, hi[2] = {0.f, 0.f};
    for (int kb = warp; kb < KB; kb += 8) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            float v[32];
            load(row0 + 8 * h, kb, v);
#pragma unroll
            for (int i = 0; i < 32; ++i) { lo[h] = fminf(lo[h], v[i]); hi[h] = fmaxf(hi[h], v[i]); }
        }
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
#pragma unroll
        for (int d = 1; d < 4; d <<= 1) {
            lo[h] = fminf(lo[h], __shfl_sync(0xffffffffu, lo[h], partner(d)));
            hi[h] = fmaxf(hi[h], __shfl_sync(0xffffffffu, hi[h], partner(d)));
        }
        if (q == 0) { s_ext[warp][0][8 * h + r] = lo[h]; s_ext[warp][1][8 * h + r] = hi[h]; }
    }
    __syncthreads();
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        for (int w = 0; w < 8; ++w) { lo[h] = fminf(lo[h], s_ext[w][0][8 * h + r]); hi[h] = fmaxf(hi[h], s_ext[w][1][8 * h + r]); }
        const float top = fmaxf(-lo[h], hi[h]);
        const GroupGrid gg = group_grid(lo[h], hi[h], top, BITS, sym);
        g[h] = rounding<BITS>(gg, top);
        const int n = row0 + 8 * h;
        if (warp == 0 && q == 0) {
            scales_pc[n] = n < N ? gg.sh : __float2half_rn(0.f);
            if (!sym) zeros_pc[n] = __float2bfloat16_rn(n < N ? (float)gg.z : 0.f);
        }
    }
    for (int kb = warp; kb < KB; kb += 8) {
        uint8_t* tile = tiles + ((size_t)nt * KB + kb) * (size_t)stride;
        float v[BLOCKS == 2 ? 2 : 1][32];
        if constexpr (BLOCKS == 2) { load(row0, kb, v[0]); load(row0 + 8, kb, v[1]); }
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int n = row0 + 8 * h, at = BLOCKS == 2 ? h : 0;
            if constexpr (BLOCKS != 2) load(n, kb, v[0]);
            uint32_t c[16], w[PieceWords<BITS>::n];
#pragma unroll
            for (int G = 0; G < 4; ++G) {
                round_chunk<BITS>(v[at] + 8 * G, g[h], sym, c + 4 * G);
                if (n >= N || kb * 128 + 32 * G + 8 * q >= K) c[4 * G] = c[4 * G + 1] = c[4 * G + 2] = c[4 * G + 3] = 0u;
            }
            encode_pairs<BITS>(c, w);
            store_piece<BITS>(tile + nb * moqe_blob_bytes(BITS), h, lane, w);
        }
    }
}

// canonical [N][G] fp16 scales / zero-points out of the per-tile (or per-channel) device copies, by one thread each
struct MetaExport {
    const __half* scales_pc;
    const __nv_bfloat16* zeros_pc;
    uint16_t *scales_out, *zeros_out;       // either may be nullptr
    int G, group, sym;
};
__device__ __forceinline__ void meta_export(const uint8_t* tiles, const MetaExport& x, int N, int KB, int bits, long long i) {
    if (i >= (long long)N * x.G) return;
    const int n = (int)(i / x.G), gi = (int)(i % x.G);
    MetaSlot m = meta_slot(const_cast<uint8_t*>(tiles), const_cast<__half*>(x.scales_pc), const_cast<__nv_bfloat16*>(x.zeros_pc), bits,
                           x.group, !x.sym, KB, n, gi, 0);
    if (x.scales_out) x.scales_out[i] = __half_as_ushort(*m.s);
    if (x.zeros_out) {
        const float z = x.sym ? (float)(1 << (bits - 1)) : __bfloat162float(*m.z);
        x.zeros_out[i] = __half_as_ushort(__float2half_rn(z));
    }
}

// The codes' blocks first, then those of the scales and zero-points (11008 x 4096, 4-bit g128: 14.7 us for the codes, and 5.7
// and a launch for a kernel of 1400 blocks that waits on scattered loads; together 17.7).
template <int BITS>
__global__ void unpack_kernel(const uint8_t* __restrict__ tiles, int N, int K, int KB, int tile_stride,
                              uint8_t* __restrict__ canon, long long npieces, unsigned code_blocks, const MetaExport x) {
    if (blockIdx.x >= code_blocks) {
        meta_export(tiles, x, N, KB, BITS, (long long)(blockIdx.x - code_blocks) * blockDim.x + threadIdx.x);
        return;
    }
    long long pid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (pid >= npieces) return;
    PieceCoord pc = piece_coord(pid, KB);
    if (pc.n >= N) return;
    uint32_t w[PieceWords<BITS>::n];
    load_piece<BITS>(tiles + pc.tile_index * (size_t)tile_stride + pc.nb * moqe_blob_bytes(BITS), pc.half, pc.slot, w);
    uint32_t c[32];
    decode_piece<BITS>(w, c);
#pragma unroll
    for (int G = 0; G < 4; ++G) {
        int k0 = pc.kb * 128 + 32 * G + 8 * pc.q;
        if (k0 >= K) continue;
        uint2 v;
        v.x = c[8 * G] | (c[8 * G + 1] << 8) | (c[8 * G + 2] << 16) | (c[8 * G + 3] << 24);
        v.y = c[8 * G + 4] | (c[8 * G + 5] << 8) | (c[8 * G + 6] << 16) | (c[8 * G + 7] << 24);
        *reinterpret_cast<uint2*>(canon + (size_t)pc.n * K + k0) = v;
    }
}

// canonical [N][G] fp16 scales / zero-points -> the per-tile (or per-channel) device copies
__global__ void meta_import_kernel(const uint16_t* __restrict__ scales_in, const uint16_t* __restrict__ zeros_in, int N, int G,
                                   int KB, int bits, int group, int sym, uint8_t* __restrict__ tiles,
                                   __half* __restrict__ scales_pc, __nv_bfloat16* __restrict__ zeros_pc) {
    long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= (long long)N * G) return;
    int n = (int)(i / G), gi = (int)(i % G);
    for (int c = 0; c < meta_copies(group); ++c) {
        MetaSlot m = meta_slot(tiles, scales_pc, zeros_pc, bits, group, !sym, KB, n, gi, c);
        *m.s = __ushort_as_half(scales_in[i]);
        if (!sym) *m.z = __float2bfloat16_rn(__half2float(__ushort_as_half(zeros_in[i])));
    }
}

// Experts' device memory comes from a memory pool of the library's own, one per device: building an 11008 x 4096 expert
// spent 520 of its 830 us in cudaMalloc and cudaFree (the 21 experts of a LLaMA block, freed and built again: 9.8 ms; 2.5 when
// the pool kept 128 MB, 1.0 with 1 GB, which holds them).  The pool keeps at most POOL_KEEP bytes of freed memory for the next
// expert (what is above goes back to the device at the next synchronisation) and is safe for any threads and streams.  The driver
// gives that memory to allocations of the process that would fail otherwise (cudaMalloc of all free memory and 400 MB, with 830 MB
// kept here: granted); for other processes there is moqe_expert_pool_trim.
// Experts that stay make the pool grow, and then the driver's search for physical memory decides, with either allocator: 40 experts
// built and kept, microseconds each, four runs with cudaMalloc / with the pool, 4-bit 11008 x 4096 390 - 5800 / 180 - 1800, 8-bit
// 11008 x 18944 (208 MB) 450 - 2200 / 1270 - 5000.
constexpr uint64_t POOL_KEEP = 1024ull << 20;
std::mutex g_pool_mutex;
cudaMemPool_t g_pools[64] = {nullptr};
void* g_anchors[64] = {nullptr};      // a small allocation that stays: it keeps the page that device_idle takes its own from

cudaMemPool_t expert_pool(int device) {
    if (device < 0 || device >= 64) return nullptr;
    std::lock_guard<std::mutex> lock(g_pool_mutex);
    if (!g_pools[device]) {
        cudaMemPoolProps props = {};
        props.allocType = cudaMemAllocationTypePinned;
        props.location.type = cudaMemLocationTypeDevice;
        props.location.id = device;
        cudaMemPool_t pool = nullptr;
        if (cudaMemPoolCreate(&pool, &props) != cudaSuccess) { cudaGetLastError(); return nullptr; }
        uint64_t keep = POOL_KEEP;
        cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &keep);
        g_pools[device] = pool;
        if (cudaMalloc(&g_anchors[device], 4) != cudaSuccess) cudaGetLastError();
    }
    return g_pools[device];
}

// Memory for an expert that is filled on `st`, or nullptr.  A stream that is being captured gets memory from cudaMalloc, where the
// capture's mode allows it: the pool's would belong to the graph.
void* expert_malloc(size_t bytes, int device, cudaStream_t st, bool& pooled) {
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    void* p = nullptr;
    if (cudaStreamIsCapturing(st, &cap) != cudaSuccess) { cudaGetLastError(); return nullptr; }
    pooled = cap == cudaStreamCaptureStatusNone;
    cudaMemPool_t pool = pooled ? expert_pool(device) : nullptr;
    if (pooled ? !pool || cudaMallocFromPoolAsync(&p, bytes, pool, st) != cudaSuccess : cudaMalloc(&p, bytes) != cudaSuccess) {
        cudaGetLastError();
        return nullptr;
    }
    return p;
}
// Waits until the current device has done all that was enqueued on it.  By giving back a small allocation, for which cudaFree
// waits as it did when experts' own memory was given back with it: cudaDeviceSynchronize makes every capture in the process
// invalid, cudaFree none that another thread (or, in relaxed mode, this one) has under way.  5 us on an idle device; 700
// without the anchor.
bool device_idle() {
    void* p = nullptr;
    if (cudaMalloc(&p, 4) != cudaSuccess) return false;
    return cudaFree(p) == cudaSuccess;
}
// Gives it back once nothing on the device can be using it any more.
bool expert_free(void* p, bool pooled, int device) {
    int now = 0;
    if (cudaGetDevice(&now) != cudaSuccess) return false;
    bool ok = now == device || cudaSetDevice(device) == cudaSuccess;
    ok = ok && (pooled ? device_idle() && cudaFreeAsync(p, nullptr) == cudaSuccess : cudaFree(p) == cudaSuccess);
    if (!ok) cudaGetLastError();
    if (now != device) ok = cudaSetDevice(now) == cudaSuccess && ok;
    return ok;
}

moqe_status check_format(int N, int K, int bits, int group) {
    if (N <= 0 || K <= 0) return MOQE_ERR_SHAPE;
    if (bits != 2 && bits != 3 && bits != 4 && bits != 8) return MOQE_ERR_UNSUPPORTED;
    if (K % 8 != 0) return MOQE_ERR_UNSUPPORTED;
    if (group < 0) return MOQE_ERR_SHAPE;
    if (group != 0) {
        if (K % group != 0) return MOQE_ERR_SHAPE;
        if (!(group == 32 || group == 64 || group % 128 == 0)) return MOQE_ERR_UNSUPPORTED;
    }
    return MOQE_OK;
}

// zeroes the buffers: padded channels / padded k have codes 0, scale 0 and zero-point 0
moqe_status clear_expert(const moqe_expert* e, cudaStream_t st) {
    return cuda_ok(cudaMemsetAsync(e->tiles, 0, e->tiles_alloc + e->pc_alloc * (e->sym ? 1 : 2), st));
}

// clear: zero the buffers on `st`; a caller that writes every byte itself does without
moqe_status alloc_expert(int N, int K, int bits, int group, int sym, bool clear, cudaStream_t st, moqe_expert** out) {
    moqe_expert* e = new (std::nothrow) moqe_expert();
    if (!e) return MOQE_ERR_ALLOC;
    e->N = N; e->K = K; e->bits = bits; e->group = group; e->sym = sym ? 1 : 0;
    e->Np = (N + 127) / 128 * 128;
    e->Kp = (K + 127) / 128 * 128;
    e->G = group ? K / group : 1;
    e->tiles = nullptr; e->scales_pc = nullptr; e->zeros_pc = nullptr;
    if (cudaGetDevice(&e->device) != cudaSuccess) { delete e; return MOQE_ERR_CUDA; }
    e->tiles_alloc = (size_t)(e->Np / 128) * (e->Kp / 128) * moqe_tile_stride(bits, group, !e->sym);
    e->pc_alloc = group == 0 ? (size_t)e->Np * 2 : 0;
    // one block: the tiles, then (per channel) scales and zero-points
    const size_t pc_total = e->pc_alloc * (e->sym ? 1 : 2);
    e->tiles = (uint8_t*)expert_malloc(e->tiles_alloc + pc_total, e->device, st, e->pooled);
    if (!e->tiles) { delete e; return MOQE_ERR_ALLOC; }
    if (group == 0) {
        e->scales_pc = (__half*)(e->tiles + e->tiles_alloc);
        if (!e->sym) e->zeros_pc = (__nv_bfloat16*)(e->tiles + e->tiles_alloc + e->pc_alloc);
    }
    if (clear && clear_expert(e, st) != MOQE_OK) { moqe_expert_destroy(e); return MOQE_ERR_CUDA; }
    *out = e;
    return MOQE_OK;
}

// Blocks of quantize_channel_kernel to an SM.  Three, unless their rows are too many for L2 (148 x 3 x 16 rows of K floats against 126
// MB: beyond some 3800 k the second pass goes to HBM) and two have no more strips after one another on an SM, or as many and a last
// round that is a good part empty either way.  Three / two, us, 8 bit and 3 bit: 11008 x 4096 111 / 105, 111 / 95; 10656 x 5120 129 / 120,
// 132 / 115; 9472 x 4096 97 / 79; 18944 x 4096 165 / 151.  But 11008 x 3584 94 / 99, 13312 x 4096 112 / 113, 21312 x 4096 168 / 183,
// 4736 x 4096 (one round) 40 / 42.
int channel_blocks(int strips, int K) {
    const int sms = device_sm_count();
    auto rounds = [&](int b) { return (strips - sms / 8 + b * sms - 1) / (b * sms) * b; };      // (a few strips more make no round)
    const int two = rounds(2), three = rounds(3);
    return K > 3840 && strips > 2 * sms && (two < three || (two == three && strips * 20ll < 17ll * sms * three)) ? 2 : 3;
}

moqe_status launch_quantize(const moqe_expert* e, const float* W, cudaStream_t st) {
    const int KB = e->Kp / 128, strips = e->Np / 16;
    if (e->group == 0) {
        const int blocks = channel_blocks(strips, e->K);
#define MOQE_QC(B) (blocks == 2 ? quantize_channel_kernel<B, 2> : quantize_channel_kernel<B, 3>)<<<strips, 256, 0, st>>>(W, e->N, e->K, e->sym, KB, e->tiles, e->scales_pc, e->zeros_pc)
        if (e->bits == 4) MOQE_QC(4);
        else if (e->bits == 8) MOQE_QC(8);
        else if (e->bits == 2) MOQE_QC(2);
        else MOQE_QC(3);
#undef MOQE_QC
        count_launch();
        return cuda_ok(cudaGetLastError());
    }
    // W[N][K]: boxes of 32 k x 16 rows, 128-byte swizzle, zero fill outside
    const EncodeTiledFn enc = encode_tiled_fn();
    int* status = device_status_word();
    if (!enc || !status) return MOQE_ERR_CUDA;
    CUtensorMap map;
    const cuuint64_t dim[2] = {(cuuint64_t)e->K, (cuuint64_t)e->N}, pitch[1] = {(cuuint64_t)e->K * 4};
    const cuuint32_t box[2] = {32, 16}, es[2] = {1, 1};
    if (enc(&map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, const_cast<float*>(W), dim, pitch, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
            CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
        return MOQE_ERR_CUDA;
    const long long blobs = (long long)strips * KB;
    const int sms = device_sm_count();
    const unsigned grid = (unsigned)(blobs < sms ? blobs : sms);
    auto run = [&](auto kernel, std::atomic<unsigned long long>& attr) {
        if (!ensure_dynamic_smem((const void*)kernel, QG_SMEM, attr)) return false;
        kernel<<<grid, QG_WARPS * 32, QG_SMEM, st>>>(map, e->N, e->K, e->group, e->sym, KB, blobs, e->tiles, status);
        return true;
    };
    static std::atomic<unsigned long long> attr[4] = {};
    if (!(e->bits == 4 ? run(quantize_group_kernel<4>, attr[0]) : e->bits == 8 ? run(quantize_group_kernel<8>, attr[1])
          : e->bits == 2 ? run(quantize_group_kernel<2>, attr[2]) : run(quantize_group_kernel<3>, attr[3]))) {
        cudaGetLastError();
        return MOQE_ERR_CUDA;
    }
    count_launch();
    return cuda_ok(cudaGetLastError());
}

// Whether an expert is built by one kernel, or by the two before them.  Groups within a k-block are.  A per-channel
// expert's strip of 16 rows belongs to one block there, which goes over it twice: that wants strips for every SM to the last
// round, and short enough to be in L2 the second time.  Two kernels / one, device time in us, 8 bit: 11008 rows (688 strips on 148
// SMs) x 4096 113 / 105, x 11008 267 / 296; 3072 rows (192 strips) x 4096 36 / 44; 128 rows x 11008 23 / 60.  Rows of up to 1024
// are over before the second launch would start (128 x 1024 18 / 12, 11008 x 1024 34 / 33).
bool one_kernel(const moqe_expert* e) {
    if (e->group != 0) return e->group <= 128;
    const int strips = e->Np / 16, sms = device_sm_count(), rounds = (strips + sms - 1) / sms;
    return e->K <= 1024 || (e->K <= 5120 && strips * 10ll >= 9ll * sms * rounds);
}

template <bool FROM_CODES>
moqe_status launch_encode(const moqe_expert* e, const float* W, const uint8_t* canon, cudaStream_t st) {
    int KB = e->Kp / 128;
    long long npieces = (long long)(e->Np / 128) * KB * 512;
    unsigned blocks = (unsigned)((npieces + 127) / 128);
#define MOQE_ENC(B)                                                                                                  \
    encode_pack_kernel<B, FROM_CODES><<<blocks, 128, 0, st>>>(W, canon, e->N, e->K, e->group, e->sym, KB, e->tiles,   \
                                                              e->scales_pc, e->zeros_pc, npieces)
    if (e->bits == 4) MOQE_ENC(4);
    else if (e->bits == 8) MOQE_ENC(8);
    else if (e->bits == 2) MOQE_ENC(2);
    else MOQE_ENC(3);
#undef MOQE_ENC
    count_launch();
    return cuda_ok(cudaGetLastError());
}

}  // namespace
}  // namespace moqe

using namespace moqe;

extern "C" moqe_status moqe_quantize_rtn(const float* W, int N, int K, int bits, int group, int sym, void* stream,
                                         moqe_expert** out) {
    if (!W || !out) return MOQE_ERR_NULL;
    moqe_status s = check_format(N, K, bits, group);
    if (s != MOQE_OK) return s;
    if (reinterpret_cast<uintptr_t>(W) % 16 != 0) return MOQE_ERR_UNSUPPORTED;
    cudaStream_t st = (cudaStream_t)stream;
    moqe_expert* e = nullptr;
    s = alloc_expert(N, K, bits, group, sym, false, st, &e);
    if (s != MOQE_OK) return s;
    if (one_kernel(e)) {                                 // (it writes every byte)
        s = launch_quantize(e, W, st);
        if (s != MOQE_OK) { moqe_expert_destroy(e); return s; }
        *out = e;
        return MOQE_OK;
    }
    if (e->N != e->Np || e->K != e->Kp) {                // (without padding the two kernels write every byte as well)
        s = clear_expert(e, st);
        if (s != MOQE_OK) { moqe_expert_destroy(e); return s; }
    }
    long long warps = (long long)N * e->G;
    unsigned blocks = (unsigned)((warps * 32 + 255) / 256);
    rtn_scales_kernel<<<blocks, 256, 0, st>>>(W, N, K, bits, group, e->G, e->sym, e->Kp / 128, e->tiles, e->scales_pc,
                                              e->zeros_pc);
    count_launch();
    if (cudaGetLastError() != cudaSuccess) { moqe_expert_destroy(e); return MOQE_ERR_CUDA; }
    s = launch_encode<false>(e, W, nullptr, st);
    if (s != MOQE_OK) { moqe_expert_destroy(e); return s; }
    *out = e;
    return MOQE_OK;
}

extern "C" moqe_status moqe_expert_import(int N, int K, int bits, int group, int sym, const uint8_t* codes,
                                          const uint16_t* scales_f16, const uint16_t* zeros_f16, void* stream,
                                          moqe_expert** out) {
    if (!codes || !scales_f16 || !out) return MOQE_ERR_NULL;
    if (!sym && !zeros_f16) return MOQE_ERR_NULL;
    moqe_status s = check_format(N, K, bits, group);
    if (s != MOQE_OK) return s;
    if (reinterpret_cast<uintptr_t>(codes) % 8 != 0) return MOQE_ERR_UNSUPPORTED;
    cudaStream_t st = (cudaStream_t)stream;
    moqe_expert* e = nullptr;
    s = alloc_expert(N, K, bits, group, sym, true, st, &e);
    if (s != MOQE_OK) return s;
    long long n = (long long)N * e->G;
    meta_import_kernel<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(scales_f16, zeros_f16, N, e->G, e->Kp / 128, bits, group,
                                                                    e->sym, e->tiles, e->scales_pc, e->zeros_pc);
    count_launch();
    if (cudaGetLastError() != cudaSuccess) { moqe_expert_destroy(e); return MOQE_ERR_CUDA; }
    s = launch_encode<true>(e, nullptr, codes, st);
    if (s != MOQE_OK) { moqe_expert_destroy(e); return s; }
    *out = e;
    return MOQE_OK;
}

extern "C" moqe_status moqe_expert_export(const moqe_expert* e, uint8_t* codes, uint16_t* scales_f16,
                                          uint16_t* zeros_f16, void* stream) {
    if (!e) return MOQE_ERR_NULL;
    cudaStream_t st = (cudaStream_t)stream;
    if (codes && reinterpret_cast<uintptr_t>(codes) % 8 != 0) return MOQE_ERR_UNSUPPORTED;
    const int KB = e->Kp / 128, stride = moqe_tile_stride(e->bits, e->group, !e->sym);
    const long long npieces = codes ? (long long)(e->Np / 128) * KB * 512 : 0;
    const unsigned code_blocks = (unsigned)((npieces + 127) / 128);
    const bool meta = scales_f16 || zeros_f16;
    const unsigned blocks = code_blocks + (meta ? (unsigned)(((long long)e->N * e->G + 127) / 128) : 0u);
    const MetaExport x = {e->scales_pc, e->zeros_pc, scales_f16, zeros_f16, e->G, e->group, e->sym};
    if (blocks > 0) {
        if (e->bits == 4) unpack_kernel<4><<<blocks, 128, 0, st>>>(e->tiles, e->N, e->K, KB, stride, codes, npieces, code_blocks, x);
        else if (e->bits == 8) unpack_kernel<8><<<blocks, 128, 0, st>>>(e->tiles, e->N, e->K, KB, stride, codes, npieces, code_blocks, x);
        else if (e->bits == 2) unpack_kernel<2><<<blocks, 128, 0, st>>>(e->tiles, e->N, e->K, KB, stride, codes, npieces, code_blocks, x);
        else unpack_kernel<3><<<blocks, 128, 0, st>>>(e->tiles, e->N, e->K, KB, stride, codes, npieces, code_blocks, x);
        count_launch();
    }
    return cuda_ok(cudaGetLastError());
}

extern "C" moqe_status moqe_expert_info(const moqe_expert* e, int* N, int* K, int* bits, int* group, int* sym,
                                        size_t* code_bytes, size_t* meta_bytes, size_t* alloc_bytes) {
    if (!e) return MOQE_ERR_NULL;
    if (N) *N = e->N;
    if (K) *K = e->K;
    if (bits) *bits = e->bits;
    if (group) *group = e->group;
    if (sym) *sym = e->sym;
    if (code_bytes) *code_bytes = (size_t)e->N * e->K * e->bits / 8;
    if (meta_bytes) *meta_bytes = (size_t)e->N * e->G * 2 * (e->sym ? 1 : 2);
    if (alloc_bytes) *alloc_bytes = e->tiles_alloc + e->pc_alloc * (e->sym ? 1 : 2);
    return MOQE_OK;
}

extern "C" moqe_status moqe_expert_pool_trim(size_t keep_bytes) {
    int device = 0;
    if (cudaGetDevice(&device) != cudaSuccess) return MOQE_ERR_CUDA;
    cudaMemPool_t pool = expert_pool(device);
    if (!pool) return MOQE_ERR_ALLOC;
    // (the last experts were given back on the default stream)
    return cuda_ok(cudaStreamSynchronize(nullptr) != cudaSuccess ? cudaGetLastError() : cudaMemPoolTrimTo(pool, keep_bytes));
}

extern "C" moqe_status moqe_expert_destroy(moqe_expert* e) {
    if (!e) return MOQE_ERR_NULL;
    const bool ok = expert_free(e->tiles, e->pooled, e->device);
    delete e;
    return ok ? MOQE_OK : MOQE_ERR_CUDA;
}

// ---------------------------------------------------------------------------- dense copy of a small expert
// For layers whose weights are a few hundred kilobytes (1x1 convolutions) the routed product is bound by the
// activations, and the weights are best handed to the tensor cores as a plain bf16 matrix Wd[Np][Kp] (row = output
// channel, K contiguous).  Per-channel experts: Wd = c - z, an exact small integer, and col_scale[n] = the channel's
// scale, applied to the fp32 sums.  Grouped experts: s * (c - z) (exact in fp32) is split into two bf16 numbers,
// hi = bf16(w) in columns [0, Kp) and lo = bf16(w - hi) in columns [Kp, 2 Kp), and col_scale[n] = 1: the caller
// multiplies the activations by both halves, which leaves a relative error of 2^-17 per weight.  Rows are 2 Kp wide.
namespace moqe {
namespace {
struct DenseSrc {
    const uint8_t* tiles[MOQE_MAX_EXPERTS];
    const __half* scales_pc[MOQE_MAX_EXPERTS];
    const __nv_bfloat16* zeros_pc[MOQE_MAX_EXPERTS];
    int bits[MOQE_MAX_EXPERTS], group[MOQE_MAX_EXPERTS], sym[MOQE_MAX_EXPERTS];
};

template <int BITS>
__device__ __forceinline__ void dense_unpack_piece(const uint8_t* __restrict__ tiles, const __half* __restrict__ scales_pc,
                                                   const __nv_bfloat16* __restrict__ zeros_pc, int N, int K, int Kp, int KB, int group,
                                                   int sym, uint16_t* __restrict__ Wd, float* __restrict__ col_scale, long long pid) {
    PieceCoord pc = piece_coord(pid, KB);
    const int stride = moqe_tile_stride(BITS, group, !sym);
    uint32_t w[PieceWords<BITS>::n];
    load_piece<BITS>(tiles + pc.tile_index * (size_t)stride + pc.nb * moqe_blob_bytes(BITS), pc.half, pc.slot, w);
    uint32_t c[32];
    decode_piece<BITS>(w, c);
    const bool live = pc.n < N;
    if (pc.kb == 0 && pc.q == 0) col_scale[pc.n] = !live ? 0.f : (group == 0 ? __half2float(scales_pc[pc.n]) : 1.f);
#pragma unroll
    for (int G = 0; G < 4; ++G) {
        const int k0 = pc.kb * 128 + 32 * G + 8 * pc.q;
        uint32_t o[4] = {0u, 0u, 0u, 0u}, o2[4] = {0u, 0u, 0u, 0u};
        if (live && k0 < K) {
            float s = 1.f, z = (float)(1 << (BITS - 1));
            if (group == 0) {
                if (!sym) z = __bfloat162float(zeros_pc[pc.n]);
            } else {
                MetaSlot m = meta_slot(const_cast<uint8_t*>(tiles), nullptr, nullptr, BITS, group, !sym, KB, pc.n, k0 / group, 0);
                s = __half2float(*m.s);
                if (!sym) z = __bfloat162float(*m.z);
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float w0 = s * ((float)c[8 * G + 2 * i] - z), w1 = s * ((float)c[8 * G + 2 * i + 1] - z);
                __nv_bfloat162 v = __floats2bfloat162_rn(w0, w1);
                o[i] = *reinterpret_cast<uint32_t*>(&v);
                if (group != 0) {
                    __nv_bfloat162 r = __floats2bfloat162_rn(w0 - __low2float(v), w1 - __high2float(v));
                    o2[i] = *reinterpret_cast<uint32_t*>(&r);
                }
            }
        }
        *reinterpret_cast<uint4*>(Wd + (size_t)pc.n * 2 * Kp + k0) = make_uint4(o[0], o[1], o[2], o[3]);
        *reinterpret_cast<uint4*>(Wd + (size_t)pc.n * 2 * Kp + Kp + k0) = make_uint4(o2[0], o2[1], o2[2], o2[3]);
    }
}

// blockIdx.y = expert
__global__ void dense_unpack_kernel(const __grid_constant__ DenseSrc src, int N, int K, int Np, int Kp, int KB,
                                    uint16_t* __restrict__ Wd, float* __restrict__ col_scale, long long npieces) {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");     // (the GEMM behind may start its prologue)
    const long long pid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (pid >= npieces) return;
    const int e = blockIdx.y;
    uint16_t* wd = Wd + (size_t)e * Np * 2 * Kp;
    float* cs = col_scale + (size_t)e * Np;
    if (src.bits[e] == 4) dense_unpack_piece<4>(src.tiles[e], src.scales_pc[e], src.zeros_pc[e], N, K, Kp, KB, src.group[e], src.sym[e], wd, cs, pid);
    else if (src.bits[e] == 8) dense_unpack_piece<8>(src.tiles[e], src.scales_pc[e], src.zeros_pc[e], N, K, Kp, KB, src.group[e], src.sym[e], wd, cs, pid);
    else if (src.bits[e] == 2) dense_unpack_piece<2>(src.tiles[e], src.scales_pc[e], src.zeros_pc[e], N, K, Kp, KB, src.group[e], src.sym[e], wd, cs, pid);
    else dense_unpack_piece<3>(src.tiles[e], src.scales_pc[e], src.zeros_pc[e], N, K, Kp, KB, src.group[e], src.sym[e], wd, cs, pid);
}
}  // namespace

moqe_status launch_dense_unpack(const moqe_expert* const* ex, int E, uint16_t* Wd, float* col_scale, cudaStream_t st) {
    DenseSrc src;
    for (int e = 0; e < E; ++e) {
        src.tiles[e] = ex[e]->tiles; src.scales_pc[e] = ex[e]->scales_pc; src.zeros_pc[e] = ex[e]->zeros_pc;
        src.bits[e] = ex[e]->bits; src.group[e] = ex[e]->group; src.sym[e] = ex[e]->sym;
    }
    const int KB = ex[0]->Kp / 128;
    const long long npieces = (long long)(ex[0]->Np / 128) * KB * 512;
    dense_unpack_kernel<<<dim3((unsigned)((npieces + 127) / 128), E), 128, 0, st>>>(src, ex[0]->N, ex[0]->K, ex[0]->Np, ex[0]->Kp, KB, Wd,
                                                                                  col_scale, npieces);
    count_launch();
    return cuda_ok(cudaGetLastError());
}
}  // namespace moqe

// ---------------------------------------------------------------------------- expert residency
// Section 4.4 of the paper and its appendix table "Router model and expert loading overhead": one expert is kept on
// the GPU, the others wait in CPU RAM (or on disk) and are loaded when the routing changes.  A packed expert is a
// plain byte image (its tiles, and for per-channel experts the scale / zero-point arrays), so moving it is pure
// copy-engine work: to a file, to pinned host memory, and back on a side stream while the current layer runs.
namespace moqe {
namespace {

struct ImageHeader {
    char magic[8];                 // "MOQEXP1\0"
    int32_t layout;                // version of the packed layout this library writes
    int32_t N, K, bits, group, sym;
    uint64_t tiles_bytes, pc_bytes;
};
constexpr int32_t PACKED_LAYOUT_VERSION = 1;

ImageHeader header_of(const moqe_expert* e) {
    ImageHeader h = {};
    memcpy(h.magic, "MOQEXP1", 8);
    h.layout = PACKED_LAYOUT_VERSION;
    h.N = e->N; h.K = e->K; h.bits = e->bits; h.group = e->group; h.sym = e->sym;
    h.tiles_bytes = e->tiles_alloc; h.pc_bytes = e->pc_alloc;
    return h;
}
// does the header describe an expert this library would lay out in exactly these sizes?
moqe_status header_ok(const ImageHeader& h) {
    if (memcmp(h.magic, "MOQEXP1", 8) != 0 || h.layout != PACKED_LAYOUT_VERSION) return MOQE_ERR_UNSUPPORTED;
    moqe_status s = check_format(h.N, h.K, h.bits, h.group);
    if (s != MOQE_OK) return s;
    const size_t Np = (size_t)(h.N + 127) / 128 * 128, Kp = (size_t)(h.K + 127) / 128 * 128;
    const size_t tiles = (Np / 128) * (Kp / 128) * moqe_tile_stride(h.bits, h.group, !h.sym);
    const size_t pc = h.group == 0 ? Np * 2 : 0;
    return (h.tiles_bytes == tiles && h.pc_bytes == pc && (h.sym == 0 || h.sym == 1)) ? MOQE_OK : MOQE_ERR_SHAPE;
}
size_t image_bytes(const ImageHeader& h) { return (size_t)h.tiles_bytes + (size_t)h.pc_bytes * (h.sym ? 1 : 2); }

}  // namespace
}  // namespace moqe

// A packed expert parked in pinned host memory: header + byte image.
struct moqe_expert_host {
    moqe::ImageHeader h;
    uint8_t* image;                // pinned: tiles, then scales_pc, then zeros_pc
};

extern "C" moqe_status moqe_expert_offload(const moqe_expert* e, void* stream, moqe_expert_host** out) {
    if (!e || !out) return MOQE_ERR_NULL;
    moqe_expert_host* hx = new (std::nothrow) moqe_expert_host();
    if (!hx) return MOQE_ERR_ALLOC;
    hx->h = header_of(e);
    hx->image = nullptr;
    if (cudaMallocHost(&hx->image, image_bytes(hx->h)) != cudaSuccess) { cudaGetLastError(); delete hx; return MOQE_ERR_ALLOC; }
    cudaStream_t st = (cudaStream_t)stream;
    cudaError_t err = cudaMemcpyAsync(hx->image, e->tiles, e->tiles_alloc, cudaMemcpyDeviceToHost, st);
    if (err == cudaSuccess && e->scales_pc) err = cudaMemcpyAsync(hx->image + e->tiles_alloc, e->scales_pc, e->pc_alloc, cudaMemcpyDeviceToHost, st);
    if (err == cudaSuccess && e->zeros_pc) err = cudaMemcpyAsync(hx->image + e->tiles_alloc + e->pc_alloc, e->zeros_pc, e->pc_alloc, cudaMemcpyDeviceToHost, st);
    if (err == cudaSuccess) err = cudaStreamSynchronize(st);       // the image is complete when the call returns
    if (err != cudaSuccess) { cudaFreeHost(hx->image); delete hx; return MOQE_ERR_CUDA; }
    *out = hx;
    return MOQE_OK;
}

extern "C" moqe_status moqe_expert_prefetch(const moqe_expert_host* hx, void* stream, moqe_expert** out) {
    if (!hx || !out) return MOQE_ERR_NULL;
    moqe_status s = header_ok(hx->h);
    if (s != MOQE_OK) return s;
    cudaStream_t st = (cudaStream_t)stream;
    moqe_expert* e = nullptr;
    s = alloc_expert(hx->h.N, hx->h.K, hx->h.bits, hx->h.group, hx->h.sym, false, st, &e);
    if (s != MOQE_OK) return s;
    cudaError_t err = cudaMemcpyAsync(e->tiles, hx->image, e->tiles_alloc, cudaMemcpyHostToDevice, st);
    if (err == cudaSuccess && e->scales_pc) err = cudaMemcpyAsync(e->scales_pc, hx->image + e->tiles_alloc, e->pc_alloc, cudaMemcpyHostToDevice, st);
    if (err == cudaSuccess && e->zeros_pc) err = cudaMemcpyAsync(e->zeros_pc, hx->image + e->tiles_alloc + e->pc_alloc, e->pc_alloc, cudaMemcpyHostToDevice, st);
    if (err != cudaSuccess) { moqe_expert_destroy(e); return MOQE_ERR_CUDA; }
    *out = e;
    return MOQE_OK;
}

extern "C" moqe_status moqe_expert_host_info(const moqe_expert_host* hx, int* N, int* K, int* bits, int* group, int* sym,
                                             size_t* image_bytes_out) {
    if (!hx) return MOQE_ERR_NULL;
    if (N) *N = hx->h.N;
    if (K) *K = hx->h.K;
    if (bits) *bits = hx->h.bits;
    if (group) *group = hx->h.group;
    if (sym) *sym = hx->h.sym;
    if (image_bytes_out) *image_bytes_out = image_bytes(hx->h);
    return MOQE_OK;
}

extern "C" moqe_status moqe_expert_host_destroy(moqe_expert_host* hx) {
    if (!hx) return MOQE_ERR_NULL;
    cudaError_t a = cudaFreeHost(hx->image);
    delete hx;
    return a == cudaSuccess ? MOQE_OK : MOQE_ERR_CUDA;
}

extern "C" moqe_status moqe_expert_host_save(const moqe_expert_host* hx, const char* path) {
    if (!hx || !path) return MOQE_ERR_NULL;
    FILE* f = fopen(path, "wb");
    if (!f) return MOQE_ERR_IO;
    const size_t n = image_bytes(hx->h);
    const bool ok = fwrite(&hx->h, sizeof(hx->h), 1, f) == 1 && (n == 0 || fwrite(hx->image, 1, n, f) == n);
    const bool closed = fclose(f) == 0;
    return ok && closed ? MOQE_OK : MOQE_ERR_IO;
}

extern "C" moqe_status moqe_expert_host_load(const char* path, moqe_expert_host** out) {
    if (!path || !out) return MOQE_ERR_NULL;
    FILE* f = fopen(path, "rb");
    if (!f) return MOQE_ERR_IO;
    ImageHeader h;
    if (fread(&h, sizeof(h), 1, f) != 1) { fclose(f); return MOQE_ERR_IO; }
    moqe_status s = header_ok(h);
    if (s != MOQE_OK) { fclose(f); return s; }
    // the file must hold exactly the image the header promises
    const size_t n = image_bytes(h);
    if (fseek(f, 0, SEEK_END) != 0 || (size_t)ftell(f) != sizeof(h) + n || fseek(f, (long)sizeof(h), SEEK_SET) != 0) { fclose(f); return MOQE_ERR_IO; }
    moqe_expert_host* hx = new (std::nothrow) moqe_expert_host();
    if (!hx) { fclose(f); return MOQE_ERR_ALLOC; }
    hx->h = h;
    hx->image = nullptr;
    if (cudaMallocHost(&hx->image, n ? n : 1) != cudaSuccess) { cudaGetLastError(); delete hx; fclose(f); return MOQE_ERR_ALLOC; }
    const bool ok = fread(hx->image, 1, n, f) == n;
    fclose(f);
    if (!ok) { cudaFreeHost(hx->image); delete hx; return MOQE_ERR_IO; }
    *out = hx;
    return MOQE_OK;
}
