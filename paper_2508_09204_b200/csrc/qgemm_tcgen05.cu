// Routed dequant-GEMM for batches beyond the decode kernel's: a persistent, warp-specialised grouped GEMM on the
// 5th-generation tensor cores, two SMs to a tile (cta_group::2).
//
//   tile         : 256 output channels x up to TN = 256, 128 or 64 tokens, in NH half tiles of HC = TN / NH columns.  CTA r
//                  of the pair owns channels 128 r .. 128 r + 127 (its TMEM lanes) of every token of the tile.
//   A operand    : the expert's weights, in TENSOR MEMORY.  Packed 128x128-code tiles arrive by bulk async copy; a
//                  "dequant" thread owns one channel, unpacks its 128 codes of a k-block in registers to the exact
//                  numbers (c - z) * 2^-13 in bf16 and stores them to its TMEM lane.  The unpacked weights never pass
//                  through shared memory, whose bandwidth the token operand needs.
//   B operand    : token rows, HC / 2 per CTA and half tile (each SM of the pair reads its own half and they share it).
//                  Where all of a piece's rows are consecutive in X they come in TMA boxes, one per half tile; else they are
//                  gathered through `perm` by two warps' 16-byte cp.async copies into the same swizzled layout (the fused
//                  permutation: no gathered copy of X exists).
//   accumulation : fp32 in three rotating TMEM buffers of HC tokens.  Grouped experts finish a buffer per (half tile,
//                  quantization group, at most 128 k); eight "epilogue" warps drain it, multiply by the group's fp32
//                  scale and add into register accumulators while the tensor core fills the next one:
//                      Y[m][n] = sum_G s[n][G] * (sum_{k in G} X[m][k] * (c[n][k] - z[n][G]))
//                  so the tensor core only multiplies exactly representable numbers.  Per-channel experts keep one
//                  buffer per half tile for the whole of K.
//   scheduling   : the tile list (expert, token tile, channel pair) is derived on the device from the per-expert offset
//                  table.  Whole rounds of it go tile by tile to the clusters; the rest (everything, for a small
//                  batch) is split by k-blocks ("stream-K": equal cost per cluster, whatever the routing).  A warp that
//                  holds part of a tile parks its fp32 sums and bumps an arrival counter; the last arrival adds them up
//                  in cluster order and stores.  Nobody waits for another cluster.  Rows go straight to their original
//                  positions through `perm` (fused un-permutation).
//
// Every mbarrier wait is bounded (2 s of %globaltimer); on expiry the CTA sets an abort flag, latches
// MOQE_ERR_TIMEOUT, lets copies in flight land, frees its TMEM and returns.
//
// The operation is Section 3.1 of the paper (the selected quantization expert runs the sample); the paper describes
// no kernel.
#include <cuda.h>

#include <type_traits>

#include "dequant.cuh"
#include "ptx.cuh"
#include "tc_ptx.cuh"

namespace moqe {
namespace {

constexpr int TC_MAX_CLUSTERS = 80;
constexpr int TC_EPI = 8;                          // epilogue warps
constexpr int TC_NW_MAX = 12;                      // packed-weight stages
constexpr int TC_A_COLS = 64;                      // TMEM columns of one k-block of unpacked weights
constexpr int TC_COST_MAX = 107;                   // of a k-block (kblock_cost)
// Whether the split by k-blocks may work in 32 bits.  It multiplies costs by clusters, and splits at most one tile less than there
// are clusters.
constexpr bool tc_split_fits(int clusters, int KB) { return (long long)clusters * ((long long)(clusters - 1) * KB + 1) * TC_COST_MAX < 1ll << 31; }
static_assert(tc_split_fits(74, 3715) && !tc_split_fits(74, 3768) && !tc_split_fits(TC_MAX_CLUSTERS, 4096), "74 * 73 * 3768 * 107 > 2^31");

// TN: tokens of a tile.  256: the tensor core's 1024 cycles a k-block hide one dequant warpgroup's work; 128 and 64: small
// batches, where unpacking is the critical role and gets two warpgroups.  With 64 tokens every hand-over between the roles
// costs more than the work handed over, so a step takes KS = 2 k-blocks: the two dequant groups unpack one each, the two
// epilogue groups drain one each.
template <int TN>
struct TcCfg {
    static constexpr int NH = TN == 256 ? 2 : 1;                             // half tiles
    static constexpr int KS = TN == 64 ? 2 : 1;                              // k-blocks of a step
    static constexpr int HC = TN / NH;                                       // columns of a half tile = of an accumulator buffer
    static constexpr int XR = HC / 2;                                        // token rows a CTA fetches for a half tile
    static constexpr int xhalf = 2 * XR * 128;                               // XR rows x 128 k bf16: two 64-k swizzled sub-tiles
    static constexpr int NACC = TN == 64 ? 4 : 3;                            // accumulator buffers
    static constexpr int a_base = NACC * HC;                                 // the weight buffers sit behind them
    static constexpr int NA = 2;                                             // weight buffers (of KS k-blocks)
    static_assert(a_base + NA * KS * TC_A_COLS <= 512, "tensor memory");
    static constexpr int EC = TN / 2;                                        // columns an epilogue warp stores
    static constexpr int DC = TN == 64 ? 64 : EC;                            // columns it drains
    static constexpr int dq_warps = TN == 256 ? 4 : 8;
    static constexpr int dq_arrive = KS == 2 ? 8 : 4;                        // dequant warps that fill one weight buffer
    static constexpr int epi_warp0 = 4 + dq_warps;
    static constexpr int threads = (epi_warp0 + TC_EPI) * 32;
    // registers: what the producers and the dequant warps can do without goes to the epilogue (300 rows in 128-token tiles, 4-bit g64:
    // 34 us with this split, 39 with 48 / 80 / 136; 256 tokens: with 48 / 80 / 192 the gathering producers lose more than the
    // epilogue gains, 500 scattered rows x 4096 x 4096 36.4 us and not 34.0).  The epilogue still spills, 150 bytes of the
    // 256-token tile and 60 to 80 of the others: state of the walk and loop counters, no sums.  Fewer spills were not always faster:
    // where they fall decides, and how they meet the gathers' copies, which go through the same pipe.
    static constexpr int regs_prod = TN == 256 ? 64 : (TN == 128 ? 56 : 48), regs_dq = 80, regs_epi = TN == 256 ? 184 : (TN == 128 ? 128 : 136);
    static constexpr int regs_launch = TN == 256 ? 128 : 96;
    static_assert(4 * regs_prod + dq_warps * regs_dq + TC_EPI * regs_epi <= threads / 32 * regs_launch, "setmaxnreg.inc draws on what the block was launched with");
    static constexpr int nx = 4;                                             // token stages: one step of the tile
    // (nx and NA are powers of two: stage and parity follow from the step's number)
    static_assert(NA <= nx, "the dequant warps wait for the step NA ago on its token stage's barrier");
    static constexpr int xstage = KS * NH * xhalf;
    // dynamic shared memory: token stages, packed-weight ring (a power of two of alignment slack in front)
    static constexpr int w_off = nx * xstage;
    static constexpr int n_bars = 2 * TC_NW_MAX + 2 * nx + NA + 3 * NACC + 2 * TC_EPI;   // wfull wempty xfull done afull accfull[2] accempty xchg[2]
    static constexpr int xchg_bytes = TN == 64 ? TC_EPI * 32 * 32 * 4 : 16;
    static constexpr int static_bytes = 1024 + 1600 + n_bars * 8 + TC_EPI * EC * 4 + 2 * NH * XR * 4 + 64;   // (an upper bound of TcShared)
    static constexpr int xchg_off = (227 * 1024 - static_bytes - 1024 - xchg_bytes) / 128 * 128;
    static constexpr int w_bytes = (xchg_off - w_off) / 128 * 128;
    static constexpr int dyn_bytes = 1024 + xchg_off + xchg_bytes;
};
static_assert(TcCfg<256>::w_bytes >= 3 * 18432, "shared memory budget");

struct TcParams {
    ExpertDev ex[MOQE_MAX_EXPERTS];
    const int32_t* perm;
    const int32_t* offsets;
    const uint16_t* X;
    uint16_t* Y;
    float* partials;          // [cluster][2][rank][cols / 4][128][4]
    uint32_t* counters;       // [cluster][rank][warp]; zero on entry, left zero
    int* status;
    int M, N, K, KB, E, NT1, NTP;    // NT1: 128-channel tiles, NTP: pairs of them
    int cols;                 // token columns of a parked partial sum
    int nw, wstage;           // packed-weight ring
    int split;                // 0: whole tiles only
};

// A whole warp's bounded wait.  The outcome is per lane (false: the CTA is aborting); the loops vote on it once a step, not
// after every wait (a vote each time made a wait that does not wait cost 85 cycles instead of 48).
__device__ __forceinline__ bool warp_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag, int* status) {
    bool ok = mbar_try_short(bar, parity);
    if (!ok) ok = mbar_wait_short(bar, parity, abort_flag, status);
    __syncwarp();
    return ok;
}

// ---------------------------------------------------------------------------- PTX of the two-CTA forms
__device__ __forceinline__ uint32_t cluster_rank() { uint32_t r; asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r)); return r; }
__device__ __forceinline__ uint32_t mapa(uint32_t addr, uint32_t rank) {
    uint32_t d;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(d) : "r"(addr), "r"(rank));
    return d;
}
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }
// (Arrivals on the other CTA's barriers order tensor-memory work and async copies only, so they need no cluster-scope
// release; with one, 16384 rows of a per-channel expert took 9.1 ms a LLaMA block instead of 4.9.)
__device__ __forceinline__ void remote_arrive(uint32_t cluster_addr, uint32_t count = 1) {
    asm volatile("mbarrier.arrive.shared::cluster.b64 _, [%0], %1;" ::"r"(cluster_addr), "r"(count) : "memory");
}
// One lane of a warp arrives.  Predicated: as a branch of one lane each of these cost the warp 100 cycles and more, several
// times a k-block (see dequant_piece).
__device__ __forceinline__ void remote_arrive_if(bool yes, uint32_t cluster_addr, uint32_t count = 1) {
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %2, 0;\n\t@p mbarrier.arrive.shared::cluster.b64 _, [%0], %1;\n\t}"
                 ::"r"(cluster_addr), "r"(count), "r"((uint32_t)yes) : "memory");
}
__device__ __forceinline__ void remote_arrive_expect_tx(uint32_t cluster_addr, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.relaxed.cluster.shared::cluster.b64 _, [%0], %1;" ::"r"(cluster_addr), "r"(bytes) : "memory");
}
__device__ __forceinline__ void tma_box_pair(uint32_t dst, const CUtensorMap* map, int c0, int c1, uint32_t cluster_bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes.cta_group::2 [%0], [%1, {%2, %3}], [%4];"
        ::"r"(dst), "l"(map), "r"(c0), "r"(c1), "r"(cluster_bar) : "memory");
}
__device__ __forceinline__ void prefetch_tmap(const CUtensorMap* map) { asm volatile("prefetch.tensormap [%0];" ::"l"(map) : "memory"); }
__device__ __forceinline__ void tmem_alloc_pair(uint32_t smem_dst, uint32_t cols) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_dst), "r"(cols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc_pair(uint32_t taddr, uint32_t cols) {
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(cols) : "memory");
}
// D[256 x n] (+)= A[256 x 16] (TMEM of both CTAs) . B[n x 16]^T (n / 2 rows in each CTA's shared memory)
__device__ __forceinline__ void umma_pair_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t bdesc, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
        ::"r"(d_tmem), "r"(a_tmem), "l"(bdesc), "r"(idesc), "r"(accumulate) : "memory");
}
// arrives at the same barrier of both CTAs when every MMA issued so far is done
__device__ __forceinline__ void umma_commit_pair(uint32_t bar) {
    const uint16_t both = 3;
    asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(bar), "h"(both) : "memory");
}
// bf16 x bf16 -> fp32, both operands K-major, M = 256 over the pair, N = n
__device__ __forceinline__ uint32_t umma_idesc_pair(int n) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((256u >> 4) << 24);
}

// ---------------------------------------------------------------------------- schedule
// (static shared memory: every address is a constant of the code, not a register)
struct TcSched {
    int off[MOQE_MAX_EXPERTS + 1];
    int tile0[MOQE_MAX_EXPERTS + 1];        // first tile of each expert
    int rpt[MOQE_MAX_EXPERTS];              // rows per token tile
    int us[MOQE_MAX_EXPERTS];               // first unit (k-block of a tile, counted per expert) that is split
    int ub[MOQE_MAX_EXPERTS], ue[MOQE_MAX_EXPERTS];   // this cluster's share of the split units
    int w[MOQE_MAX_EXPERTS];                // cost of a unit
    int Gs, Td;                             // clusters of the split; tiles that are not split
    int base[MOQE_MAX_EXPERTS], C;          // cost before each expert's split units; total
};
template <int TN>
struct TcShared {
    using L = TcCfg<TN>;
    unsigned long long bars[L::n_bars];
    TcSched sc;
    uint32_t tmem;
    int abort;
    __align__(16) int walk[TC_EPI][12];     // per epilogue warp: what of the walk only the end of a piece asks for
    __align__(16) int perm[TC_EPI][L::EC];  // per epilogue warp: its columns' target rows
    __align__(16) int xrow[2][L::NH * L::XR];   // rows of X to gather, one list per gather warp: row 4 i + j at [j][i]
};
static_assert(sizeof(TcShared<256>) <= TcCfg<256>::static_bytes && sizeof(TcShared<128>) <= TcCfg<128>::static_bytes &&
                  sizeof(TcShared<64>) <= TcCfg<64>::static_bytes && sizeof(TcShared<64>) <= 48 * 1024, "shared memory budget");

struct TcPiece { int e, ntp, m0, rows, kb0, kb1, tile; };   // tile: inside the expert

// a walk over the pieces of work of one cluster: whole tiles first, then its share of the split
struct TcWalk {
    int t, e, u, ue;
    __device__ __forceinline__ void start(int cluster) { t = cluster; e = -1; u = ue = 0; }
    __device__ __forceinline__ bool next(const TcSched& s, const TcParams& p, int nclusters, TcPiece& pc) {
        int tile;
        if (t < s.Td) {
            int ee = 0;
            while (t >= s.tile0[ee + 1]) ++ee;
            pc.e = ee;
            tile = t - s.tile0[ee];
            pc.kb0 = 0;
            pc.kb1 = p.KB;
            t += nclusters;
        } else {
            while (u >= ue) {
                if (++e >= p.E) return false;
                u = s.ub[e];
                ue = s.ue[e];
            }
            pc.e = e;
            tile = u / p.KB;
            pc.kb0 = u - tile * p.KB;
            pc.kb1 = min(p.KB, pc.kb0 + (ue - u));
            u += pc.kb1 - pc.kb0;
        }
        const int mt = tile / p.NTP, rpt = s.rpt[pc.e], first = s.off[pc.e] + mt * rpt;
        pc.tile = tile;
        pc.ntp = tile - mt * p.NTP;
        pc.m0 = first;
        pc.rows = min(rpt, s.off[pc.e + 1] - first);
        return true;
    }
};
// Tokens of the first half tile, a multiple of 32: half of them, not as many as fit, so that the two epilogue groups have the
// same work (512 rows over three experts, 171 to a tile: 96 + 75 instead of 128 + 43).
template <int HC>
__device__ __forceinline__ int half_split(int rows) { return rows <= HC ? HC : ((rows + 1) / 2 + 31) & ~31; }
// MMA columns of half tile h of a tile with `rows` tokens
template <int HC>
__device__ __forceinline__ int half_cols(int rows, int h) {
    const int hs = half_split<HC>(rows);
    return (min(hs, rows - hs * h) + 31) & ~31;
}
// What a k-block of a tile costs a cluster, in units of 64 cycles or so: by tile size, rows of the tile and quantization groups per
// k-block.  At most TC_COST_MAX.  Decides the shares of clusters that split tiles of several formats, and what is worth splitting.
// Taken with every cluster busy; whole tiles of one format, 4 bit, take now (pc, g128, g64, g32) 20, 22, 42, 71 with 256 rows, 12, 17,
// 31, 53 with 128; 128 tokens 12, 16, 25, 48; 64 tokens 10, 12, 22, 33.  With those figures here mixed batches are as often slower
// as faster (2926 rows x 512 x 3584, W8-pc W4-g64: 35.2 instead of 31.0 us; 250 rows x 4096 x 4096, W8-pc W4-g32 W4-g128: 2.6 % less):
// shares are cut in whole k-blocks, and a gathered or parked k-block costs more than these.
template <int TN>
__device__ __forceinline__ int kblock_cost(int rows, int bits, int per) {
    const int wide = bits == 8 || bits == 3 ? 2 : 0;       // (the 8-bit tiles are larger, the 3-bit ones take longer to unpack)
    if (TN == 64) return (per <= 1 ? 13 : (per == 2 ? 22 : 36)) + wide;
    if (TN == 128) return (per == 0 ? 16 : (per == 1 ? 18 : (per == 2 ? 32 : 57))) + wide / 2;
    return (rows <= 128 ? (per == 0 ? 18 : (per == 1 ? 23 : (per == 2 ? 39 : 68))) : (per == 0 ? 22 : (per == 1 ? 23 : (per == 2 ? 50 : 106)))) + wide / 2;
}

// ---------------------------------------------------------------------------- unpacking
__device__ __forceinline__ uint32_t fma_bf16x2(uint32_t a, uint32_t b, uint32_t c) {
    const __nv_bfloat162 r = __hfma2(*reinterpret_cast<const __nv_bfloat162*>(&a), *reinterpret_cast<const __nv_bfloat162*>(&b),
                                     *reinterpret_cast<const __nv_bfloat162*>(&c));
    return *reinterpret_cast<const uint32_t*>(&r);
}
// Chunk G of a piece as bf16 pairs (c - z) * 2^-13.  A code zero-extended to 16 bits IS the bf16 number c * 2^-133
// (subnormal below 128; the encoding runs on linearly through the first normal binade, so a code may also sit up to
// four, three or six bits higher as long as it stays below bit 8).  One fused multiply-add per PAIR of codes,
// c * 2^(-133+s) * 2^(120-s) - z * 2^-13, is exact (|c - z| <= 255 has 8 significant bits); the scale takes the 2^13.
// nz: -z * 2^-13 in both halves.
template <int BITS, int G>
__device__ __forceinline__ void unpack_scaled(const uint32_t (&w)[PieceWords<BITS>::n], uint32_t nz, uint32_t* out) {
    constexpr uint32_t P120 = 0x7B807B80u, P118 = 0x7A807A80u, P117 = 0x7A007A00u, P116 = 0x79807980u, P114 = 0x78807880u;
    if constexpr (BITS == 4) {
        const uint32_t v = w[G], u = v >> 8;
        out[0] = fma_bf16x2(v & 0x000F000Fu, P120, nz);
        out[1] = fma_bf16x2(v & 0x00F000F0u, P116, nz);
        out[2] = fma_bf16x2(u & 0x000F000Fu, P120, nz);
        out[3] = fma_bf16x2(u & 0x00F000F0u, P116, nz);
    } else if constexpr (BITS == 2) {
        const uint32_t v = (G & 1) ? w[G >> 1] >> 8 : w[G >> 1];
        out[0] = fma_bf16x2(v & 0x00030003u, P120, nz);
        out[1] = fma_bf16x2(v & 0x000C000Cu, P118, nz);
        out[2] = fma_bf16x2(v & 0x00300030u, P116, nz);
        out[3] = fma_bf16x2(v & 0x00C000C0u, P114, nz);
    } else if constexpr (BITS == 3) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int p = 4 * G + i, f = p % 5;
            if (p == 15) {
                const uint32_t v = ((w[0] >> 15) & 0x00010001u) | ((w[1] >> 14) & 0x00020002u) | ((w[2] >> 13) & 0x00040004u);
                out[i] = fma_bf16x2(v, P120, nz);
            } else {
                const uint32_t v = f < 2 ? w[p / 5] : (f < 4 ? w[p / 5] >> 6 : w[p / 5] >> 12);
                out[i] = (f & 1) ? fma_bf16x2(v & 0x00380038u, P117, nz) : fma_bf16x2(v & 0x00070007u, P120, nz);
            }
        }
    } else {
#pragma unroll
        for (int i = 0; i < 4; ++i)
            out[i] = fma_bf16x2(__byte_perm(w[2 * G + (i >> 1)], 0u, (i & 1) ? 0x4342u : 0x4140u), P120, nz);
    }
}
__device__ __forceinline__ uint32_t neg_z(float z) { const float v = z * -0.0001220703125f; return pack_bf16x2(v, v); }

// The dequant role for the k-blocks of one piece.  A thread owns one channel (its TMEM lane): per k-block it reads the four
// pieces of its codes from the packed tile and fills the 64 TMEM columns of its lane.  zpc: the channel's zero-point if it
// is not in the tile (per channel, or a symmetric grid).  Returns false on abort.
// (What the loop needs of the expert is passed by value: fields of the kernel's parameters would be fetched again after
// every barrier.)
struct TcDequant {
    uint32_t bar_wfull, bar_wempty, bar_done, afull0;   // afull0: in the leading CTA
    uint32_t lane_tmem;
    int row, nw, wstage;
    uint32_t my_group;
    Ring wring;
    uint32_t step;
};
template <int TN, int BITS>
__device__ __forceinline__ bool dequant_piece(TcDequant& d, TcShared<TN>& sh, const unsigned char* wtiles, int nkb, int per,
                                              uint32_t zpc, bool tile_zeros, int* status) {
    using L = TcCfg<TN>;
    const int lane = threadIdx.x & 31, row = d.row;
    const int half = (row >> 3) & 1, r = row & 7;
    const int meta = moqe_tile_bytes(BITS) + row * 2 + 256;               // its zero-points in the tile
    const unsigned char* blobs = wtiles + (row >> 4) * moqe_blob_bytes(BITS);
    bool ok = true;
#pragma unroll 1
    for (int kb = 0; ok && kb < nkb; kb += L::KS) {
        const int nk = min(L::KS, nkb - kb);
        const int kk = L::KS == 2 ? (int)d.my_group : 0;              // this group's k-block of the step
        const bool mine = L::KS == 2 ? kk < nk : (L::dq_warps == 4 || (d.step & 1u) == d.my_group);
        if (mine) {
            if (L::KS == 2 && kk) d.wring.advance(d.nw);
            const int stage = d.wring.stage * d.wstage;
            const unsigned char* blob = blobs + stage;
            ok = warp_wait(d.bar_wfull + 8 * d.wring.stage, d.wring.phase, &sh.abort, status);
            uint32_t w[4][PieceWords<BITS>::n];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int slot = q * 8 + (r ^ (2 * q));
                if constexpr (BITS == 3) {
                    // both halves share the 16-byte slot: {A, B, C of half 0, A of half 1}
                    const uint4 v = *reinterpret_cast<const uint4*>(blob + slot * 16);
                    const uint2 u = *reinterpret_cast<const uint2*>(blob + 512 + slot * 8);
                    w[q][0] = half ? v.w : v.x;
                    w[q][1] = half ? u.x : v.y;
                    w[q][2] = half ? u.y : v.z;
                } else {
                    load_piece_smem<BITS>(blob, half, slot, w[q]);
                }
            }
            uint32_t nz[4] = {zpc, zpc, zpc, zpc};
            if (tile_zeros) {
                const unsigned char* m = wtiles + stage + meta;
                nz[0] = nz[1] = nz[2] = nz[3] = neg_z(__bfloat162float(*reinterpret_cast<const __nv_bfloat16*>(m)));
                if (per > 1) {
                    nz[3] = nz[2] = neg_z(__bfloat162float(*reinterpret_cast<const __nv_bfloat16*>(m + (per == 2 ? 1 : 2) * 512)));
                    if (per > 2) {
                        nz[1] = neg_z(__bfloat162float(*reinterpret_cast<const __nv_bfloat16*>(m + 512)));
                        nz[3] = neg_z(__bfloat162float(*reinterpret_cast<const __nv_bfloat16*>(m + 3 * 512)));
                    }
                }
            }
            // the operand buffer is free once the step NA ago is done
            if (d.step >= L::NA) ok &= warp_wait(d.bar_done + 8 * ((d.step - L::NA) % L::nx), (d.step - L::NA) / L::nx & 1u, &sh.abort, status);
            tc_fence_after();
            const uint32_t at = d.lane_tmem + (d.step % L::NA * L::KS + kk) * TC_A_COLS;
            auto chunk = [&](auto Gc) {
                constexpr int G = decltype(Gc)::value;
                uint32_t o[16];
#pragma unroll
                for (int q = 0; q < 4; ++q) unpack_scaled<BITS, G>(w[q], nz[G], o + 4 * q);
                tmem_st16(at + 16 * G, o);
            };
            chunk(std::integral_constant<int, 0>{});
            chunk(std::integral_constant<int, 1>{});
            chunk(std::integral_constant<int, 2>{});
            chunk(std::integral_constant<int, 3>{});
            // The packed tile is handed back only now that its codes have been used: an arrival right behind the loads can overtake
            // them, and the next tile may land before they are done.
            __syncwarp();
            mbar_arrive_if(lane == 0, d.bar_wempty + 8 * d.wring.stage);
            tmem_st_wait();
            tc_fence_before();
            __syncwarp();
            remote_arrive_if(lane == 0, d.afull0 + 8 * (d.step % L::NA));
            d.wring.advance(d.nw);
            if (L::KS == 2 && nk == 2 && !kk) d.wring.advance(d.nw);
            ok = __all_sync(0xffffffffu, ok);
        } else if (L::KS == 2) {
            // The step has no k-block for this group.  Its arrivals wait for the step NA ago like everyone's: earlier ones would
            // complete that step's phase in the place of a warp of the other group that has yet to store its weights.
            if (d.step >= L::NA) ok = __all_sync(0xffffffffu, warp_wait(d.bar_done + 8 * ((d.step - L::NA) % L::nx), (d.step - L::NA) / L::nx & 1u, &sh.abort, status));
            remote_arrive_if(lane == 0, d.afull0 + 8 * (d.step % L::NA));
            d.wring.advance(d.nw);
        } else {
            d.wring.advance(d.nw);
        }
        ++d.step;
    }
    return ok;
}
// the same for a CTA whose channels do not exist (the second half of the last, odd pair): the operand buffers keep whatever
// they hold (those products are never read)
template <int TN>
__device__ __forceinline__ bool dequant_none(TcDequant& d, TcShared<TN>& sh, int nkb, int* status) {
    using L = TcCfg<TN>;
    bool ok = true;
#pragma unroll 1
    for (int kb = 0; ok && kb < nkb; kb += L::KS) {
        if (L::KS == 2 || L::dq_warps == 4 || (d.step & 1u) == d.my_group) {
            if (d.step >= L::NA) ok = __all_sync(0xffffffffu, warp_wait(d.bar_done + 8 * ((d.step - L::NA) % L::nx), (d.step - L::NA) / L::nx & 1u, &sh.abort, status));
            if ((threadIdx.x & 31) == 0) remote_arrive(d.afull0 + 8 * (d.step % L::NA));
        }
        ++d.step;
    }
    return ok;
}

__device__ __forceinline__ void sts_v4(uint32_t at, int a, int b, int c, int d) {
    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(at), "r"(a), "r"(b), "r"(c), "r"(d) : "memory");
}
__device__ __forceinline__ void lds_v4(uint32_t at, int& a, int& b, int& c, int& d) {
    asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(a), "=r"(b), "=r"(c), "=r"(d) : "r"(at) : "memory");
}
// acc[0..31] += s * v, two columns per instruction (each half rounds as a scalar fma does)
__device__ __forceinline__ void fma_cols32(float* acc, const uint32_t (&v)[32], float s) {
#pragma unroll
    for (int i = 0; i < 32; i += 2)
        asm("{\n\t.reg .b64 a, x, s2;\n\tmov.b64 a, {%0, %1};\n\tmov.b64 x, {%3, %4};\n\tmov.b64 s2, {%2, %2};\n\t"
            "fma.rn.f32x2 a, s2, x, a;\n\tmov.b64 {%0, %1}, a;\n\t}"
            : "+f"(acc[i]), "+f"(acc[i + 1]) : "f"(s), "r"(v[i]), "r"(v[i + 1]));
}

// ---------------------------------------------------------------------------- the kernel
template <int TN>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(TcCfg<TN>::threads, 1)
    qgemm_tc_kernel(const __grid_constant__ TcParams p, const __grid_constant__ CUtensorMap tmap) {
    using L = TcCfg<TN>;
    constexpr int NH = L::NH, KS = L::KS, NX = L::nx, NA = L::NA, NACC = L::NACC;
    __shared__ TcShared<TN> sh;
    extern __shared__ unsigned char smem_raw[];
    unsigned char* smem = smem_raw + ((0u - smem_u32(smem_raw)) & 1023u);
    TcSched& sc = sh.sc;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t rank = cluster_rank();
    const int cluster = blockIdx.x >> 1, nclusters = gridDim.x >> 1;
    const uint32_t sbase = smem_u32(smem);
    // done[stage]: every MMA of the step in that token stage has finished.  One commit per step hands back the token
    // stage and the weight buffer and announces the accumulator buffer filled last (a commit costs the issuing warp about
    // 200 cycles, three k16 steps of a half tile).
    const uint32_t bar_wfull = smem_u32(sh.bars), bar_wempty = bar_wfull + 8 * TC_NW_MAX;
    const uint32_t bar_xfull = bar_wempty + 8 * TC_NW_MAX, bar_done = bar_xfull + 8 * NX;
    const uint32_t bar_afull = bar_done + 8 * NX;
    const uint32_t bar_accfull = bar_afull + 8 * NA, bar_accempty = bar_accfull + 16 * NACC, bar_xchg = bar_accempty + 8 * NACC;
    volatile int* s_abort = &sh.abort;

    // ---- prologue: nothing here depends on the previous kernel in the stream
    if (tid == 0) {
        for (int i = 0; i < TC_NW_MAX; ++i) { mbar_init(bar_wfull + 8 * i, 1); mbar_init(bar_wempty + 8 * i, 4); }
        for (int i = 0; i < NX; ++i) { mbar_init(bar_xfull + 8 * i, 4); mbar_init(bar_done + 8 * i, 1); }
        for (int i = 0; i < NA; ++i) mbar_init(bar_afull + 8 * i, 2 * L::dq_arrive);
        for (int i = 0; i < 2 * NACC; ++i) mbar_init(bar_accfull + 8 * i, 1);
        for (int i = 0; i < NACC; ++i) mbar_init(bar_accempty + 8 * i, 2 * TC_EPI);
        if (KS == 2)
            for (int i = 0; i < 2 * TC_EPI; ++i) mbar_init(bar_xchg + 8 * i, 1);
        *s_abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        prefetch_tmap(&tmap);
    }
    // (the pair's barriers are initialised when both CTAs have arrived here; every role waits for that before it first touches
    // the other CTA, so the round trip hides behind the schedule)
    __syncwarp();
    cluster_arrive();
    if (warp == 1) tmem_alloc_pair(smem_u32(&sh.tmem), 512);
    // ---- the schedule.  Worked out from the offset table as it stands BEFORE the previous kernel is waited for (in a block's
    // later layers it is final already), so that afterwards the table has only to be compared, while the rows of the first piece
    // are being looked up; a table that has changed is gone through again, from what the comparison has read.  (64 rows x 1024 x 1024
    // through the one-call entry point, whose sort has just written the table: 10.9 us if it is the table of the call before, 11.95 if
    // it is another; with the schedule after the wait 11.65 always.  96 rows x 4096 x 4096 on a sorted batch: 21.2, and 22.1.)
    const bool x_warp = warp == 0 || warp == 3;
    TcPiece x_pc;
    TcWalk x_wk;
    bool x_have = false;
    int x_a[NH], x_b[NH];                                  // a producer lane's rows of X: lane and lane + 32 of each half tile
    // real rows of this CTA in half tile h of a piece, and the first of them
    auto x_rows = [&](const TcPiece& pc, int h, int& first_row) {
        if (h > 0 && pc.rows <= L::HC) return 0;
        const int per_cta = half_cols<L::HC>(pc.rows, h) >> 1;
        first_row = h * half_split<L::HC>(pc.rows) + (int)rank * per_cta;
        return max(min(per_cta, pc.rows - first_row), 0);
    };
    auto x_next = [&]() {
        x_have = x_wk.next(sc, p, nclusters, x_pc);
        if (!x_have) return;
#pragma unroll
        for (int h = 0; h < NH; ++h) {
            int first_row = 0;
            const int c = x_rows(x_pc, h, first_row);
            x_a[h] = lane < c ? __ldcg(p.perm + x_pc.m0 + first_row + lane) : 0;
            x_b[h] = lane + 32 < c ? __ldcg(p.perm + x_pc.m0 + first_row + lane + 32) : 0;
        }
    };
    int t_first = 0, t_next = 0;                           // the table: its first entry, and lane e's entry e + 1
    auto read_table = [&]() {
        t_first = __ldcg(p.offsets);
        t_next = lane < p.E ? __ldcg(p.offsets + lane + 1) : 0;
    };
    auto schedule = [&]() {
        // lane e works out expert e
        const int e = lane;
        // (a table that is still being written may hold anything: offsets are made to rise and to stay within the batch)
        int o1 = min(max(t_next, 0), p.M);
        int o0 = e == 0 ? min(max(t_first, 0), p.M) : 0;
        o1 = max(o0, o1);
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int o = __shfl_up_sync(0xffffffffu, o1, d);
            if (lane >= d) o1 = max(o1, o);
        }
        {
            const int o = __shfl_up_sync(0xffffffffu, o1, 1);
            if (lane > 0) o0 = o;
        }
        const int R = o1 - o0;
        const int mt = (R + TN - 1) / TN;
        const int rpt = mt >= 4 ? TN : (mt > 0 ? ((R + mt - 1) / mt + 31) & ~31 : 32);
        const int T_e = mt * p.NTP;
        int incl = T_e;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int o = __shfl_up_sync(0xffffffffu, incl, d);
            if (lane >= d) incl += o;
        }
        const int T = __shfl_sync(0xffffffffu, incl, 31), tile0 = incl - T_e;
        const int w = e < p.E ? kblock_cost<TN>(rpt, p.ex[e].bits, moqe_groups_per_tile(p.ex[e].group)) : 1;
        // Whole rounds of tiles stay whole; what is left over is split by k-blocks if a whole tile less on the clusters that
        // would have got one is worth the parking and adding up (10 us: 16 tiles of 16 k-blocks, split, 19.9 us, whole 13.4).
        int Td = T;
        if (p.split) {
            const int left = T % nclusters;
            int wdear = mt > 0 ? w : 0;
#pragma unroll
            for (int d = 16; d > 0; d >>= 1) wdear = max(wdear, __shfl_xor_sync(0xffffffffu, wdear, d));
            if (left != 0 && (nclusters - left) * p.KB * wdear > 300 * nclusters) Td = T - left;
        }
        const int us = min(max(Td - tile0, 0), T_e) * p.KB;
        const int cnt = T_e * p.KB - us;
        const int cost = cnt * w;                          // (times the clusters within 32 bits: tc_split_fits)
        int cincl = cost;
        int wmax = cnt > 0 ? w : 1;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int o = __shfl_up_sync(0xffffffffu, cincl, d);
            if (lane >= d) cincl += o;
            wmax = max(wmax, __shfl_xor_sync(0xffffffffu, wmax, d));
        }
        const int C = __shfl_sync(0xffffffffu, cincl, 31), base = cincl - cost;
        // Every cluster's share holds at least the start of two units, and of four cheap ones: with two, few deep tiles had many
        // short pieces, and the last arrival adds them up one after another (33 rows, three experts, 256 x 8192: 24.5 -> 17.6 us,
        // where the streaming kernel takes 19.6; two experts, 256 x 11008: 31.5 -> 20.8; at worst 6 % more, 128 x 11008).  Four of
        // the dearest, groups of 32 k, are too many (9408 rows, three experts, 256 x 1024: 30.7 -> 43.3).
        const int Gs = max(1, min(nclusters, C / min(4 * wmax, max(2 * wmax, 100))));
        int ub = us, ue = us;
        if (cnt > 0 && cluster < Gs) {
            const int den = w * Gs, n0 = cluster * C - base * Gs, n1 = n0 + C;
            ub = us + min(n0 <= 0 ? 0 : (n0 + den - 1) / den, cnt);
            ue = us + min(n1 <= 0 ? 0 : (n1 + den - 1) / den, cnt);
        }
        if (e < p.E) { sc.off[e] = o0; sc.tile0[e] = tile0; }
        if (e == p.E - 1) { sc.off[p.E] = o1; sc.tile0[p.E] = T; }
        sc.rpt[e] = rpt; sc.us[e] = us; sc.ub[e] = ub; sc.ue[e] = ue; sc.w[e] = w; sc.base[e] = base;
        if (lane == 0) { sc.Gs = Gs; sc.Td = Td; sc.C = C; }
    };
#pragma unroll 1
    for (bool early = true;; early = false) {
        if (warp == 0) {
            if (early) read_table();
            schedule();
        }
        tc_fence_before();
        __syncthreads();
        bool changed = false;
        const int g_first = t_first, g_next = t_next;
        if (early) {
            if (warp == 4 && lane == 0) {
                // the first packed tiles into L2, by a warp that nobody waits for (a wrong guess costs prefetched lines only; without it 64 to
                // 96 rows of a LLaMA layer take 1 % longer)
                TcPiece pc;
                TcWalk wk;
                wk.start(cluster);
                if (wk.next(sc, p, nclusters, pc) && 2 * pc.ntp + (int)rank < p.NT1) {
                    const ExpertDev& ex = p.ex[pc.e];
                    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(ex.tiles + ((size_t)(2 * pc.ntp + (int)rank) * p.KB + pc.kb0) * ex.tile_stride),
                                 "r"(min(p.nw, pc.kb1 - pc.kb0) * ex.tile_stride) : "memory");
                }
            }
            asm volatile("griddepcontrol.wait;" ::: "memory");
            asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
        }
        if (early && warp == 0) read_table();              // (under way while the first rows are looked up)
        if (x_warp) {
            x_wk.start(cluster);
            x_next();
        }
        changed = t_first != g_first || t_next != g_next;
        if (!early || !__syncthreads_or(changed)) break;
    }
    if (warp != 2) cluster_wait();                         // (the weight producer touches its own CTA only)
    tc_fence_after();
    const uint32_t tmem_base = sh.tmem;

    if (warp < 4) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(L::regs_prod));
        if (warp == 0 || warp == 3) {
            // ---------------- X producers: this CTA's XR token rows of every half tile, KS x 128 k per stage ----------------
            // Both warps walk the stages and arrive on the pair's xfull barrier.  A piece whose rows all come in boxes has a lean
            // loop: a warp fetches one 64-k sub-tile of every box, its arrival carries the byte count, and nothing is fenced or
            // waited for (a loop for both kinds takes the warp 1170 cycles a step, more than the tensor core's 1024: 2048 rows x
            // 4096 x 4096, per channel, 57 us instead of 54).  Otherwise both warps gather, every other pair of rows each, with cp.async,
            // and the arrival for a stage follows once its copies have landed, LAG stages later, and before the next piece's rows are
            // waited for (500 scattered rows, three experts, 4096 x 4096: 33.5 us, with LAG 1 43; 481 rows in runs of 10 to 90, 4096 x
            // 11008: 67, with LAG 3 73; the stage's copies in a loop and not unrolled: 46 for the 500 rows).  TMA's own gather, four rows
            // to a request, takes an SM 45 cycles a request: 300 scattered rows 58 us and not 29.  Copies that arrive on a barrier,
            // looked at between stages, cost the other warps their issue slots: 34.
            constexpr int LAG = 2;
            const int gw = warp == 0 ? 0 : 1;
            int* s_xrow = sh.xrow[gw];
            const int hi = lane >> 4, c16 = lane & 15;
            // byte offset of this lane's 16-byte chunk of row 4 i + 2 gw + hi: sub-tile, then the 128-byte swizzle
            const uint32_t r0 = 2 * gw + hi;
            const uint32_t sw0 = (c16 >> 3) * (L::XR * 128) + r0 * 128 + (((c16 & 7) ^ r0) << 4), sw1 = (c16 >> 3) * (L::XR * 128) + (r0 + 4) * 128 + (((c16 & 7) ^ (r0 + 4)) << 4);
            uint32_t step = 0, due = 0;                    // due: the step whose arrival comes next
            bool ok = true;
            int pending = 0;
            const uint32_t full0 = mapa(bar_xfull, 0), pitch = (uint32_t)p.K * 2;
            auto arrive = [&]() {
                fence_proxy_async();
                __syncwarp();
                remote_arrive_if(lane == 0, full0 + 8 * (due % NX));
                ++due;
            };
            auto arrive_all = [&]() {
                asm volatile("cp.async.wait_group 0;" ::: "memory");
                for (; pending > 0; --pending) arrive();
            };
            for (; ok && x_have; x_next()) {
                const TcPiece pc = x_pc;
                // (the last steps of the piece before: their arrivals must not wait for this one's rows, which are being looked up)
                arrive_all();
                int src[NH], cnt[NH], boxes = 0;
                bool gathers = false;
                __syncwarp();
#pragma unroll
                for (int h = 0; h < NH; ++h) {
                    int first_row = 0;
                    const int c = x_rows(pc, h, first_row), a = x_a[h], b = x_b[h];
                    const int first = __shfl_sync(0xffffffffu, a, 0);
                    const bool run = __all_sync(0xffffffffu, (lane >= c || a == first + lane) && (lane + 32 >= c || b == first + lane + 32));
                    s_xrow[h * L::XR + (lane & 3) * (L::XR / 4) + (lane >> 2)] = a;
                    if (L::XR > 32) s_xrow[h * L::XR + (lane & 3) * (L::XR / 4) + 8 + (lane >> 2)] = b;
                    // (a box fetches XR rows whatever it needs; operand rows beyond the real ones yield columns that are
                    // never stored, so they may hold anything)
                    src[h] = c > 0 ? first : -1;
                    boxes += c > 0 ? 1 : 0;
                    cnt[h] = c;
                    gathers |= c > 0 && !(run && c > 8);
                }
                __syncwarp();
                if (!gathers) {
#pragma unroll 1
                    for (int kb0 = pc.kb0; ok && kb0 < pc.kb1; kb0 += KS, ++step) {
                        const int nk = min(KS, pc.kb1 - kb0);
                        ok = warp_wait(bar_done + 8 * (step % NX), (step / NX & 1u) ^ 1u, s_abort, p.status);
                        const uint32_t full = full0 + 8 * (step % NX);
                        if (elect_one()) {
                            remote_arrive_expect_tx(full, boxes * nk * (L::XR * 128));
#pragma unroll
                            for (int kk = 0; kk < KS; ++kk)
#pragma unroll
                                for (int h = 0; h < NH; ++h)
                                    if (kk < nk && src[h] >= 0)
                                        tma_box_pair(sbase + (step % NX) * L::xstage + (kk * NH + h) * L::xhalf + gw * (L::XR * 128), &tmap, (kb0 + kk) * 128 + gw * 64, src[h], full);
                        }
                        ok = __all_sync(0xffffffffu, ok);
                    }
                    due = step;
                    continue;
                }
#pragma unroll 1
                for (int kb0 = pc.kb0; ok && kb0 < pc.kb1; kb0 += KS) {
                    const int nk = min(KS, pc.kb1 - kb0);
                    ok = warp_wait(bar_done + 8 * (step % NX), (step / NX & 1u) ^ 1u, s_abort, p.status);
#pragma unroll
                    for (int kk = 0; kk < KS; ++kk) {
                        if (kk >= nk) break;
                        const int k = (kb0 + kk) * 128 + c16 * 8;
                        const int real = k < p.K ? 16 : 0;
                        const char* xk = reinterpret_cast<const char*>(p.X) + (real ? (size_t)k * 2 : 0);
#pragma unroll
                        for (int h = 0; h < NH; ++h) {
                            const uint32_t dst = sbase + (step % NX) * L::xstage + (kk * NH + h) * L::xhalf;
                            const int4* list = reinterpret_cast<const int4*>(s_xrow + h * L::XR + r0 * (L::XR / 4));
                            // (no branch per row: a list entry beyond the real rows is row 0, copied in vain)
#pragma unroll
                            for (int i = 0; i < L::XR / 16; ++i)
                                if (16 * i < cnt[h]) {
                                    const int4 r4 = list[i];
                                    cp_async16(dst + sw0 + i * 2048, xk + (size_t)(uint32_t)r4.x * pitch, real);
                                    cp_async16(dst + sw1 + i * 2048, xk + (size_t)(uint32_t)r4.y * pitch, real);
                                    cp_async16(dst + sw0 + i * 2048 + 1024, xk + (size_t)(uint32_t)r4.z * pitch, real);
                                    cp_async16(dst + sw1 + i * 2048 + 1024, xk + (size_t)(uint32_t)r4.w * pitch, real);
                                }
                        }
                    }
                    asm volatile("cp.async.commit_group;" ::: "memory");
                    ++step;
                    if (++pending == LAG) {
                        asm volatile("cp.async.wait_group %0;" ::"n"(LAG - 1) : "memory");
                        arrive();
                        --pending;
                    }
                    ok = __all_sync(0xffffffffu, ok);
                }
            }
            if (ok) arrive_all();
            asm volatile("cp.async.wait_group 0;" ::: "memory");
            // every stage handed back (the commits come from the leading CTA) before this CTA may exit
            for (int i = 0; ok && i < NX; ++i) {
                ok = __all_sync(0xffffffffu, mbar_wait(bar_done + 8 * (step % NX), (step / NX & 1u) ^ 1u, s_abort, p.status));
                ++step;
            }
        } else if (warp == 2) {
            // ---------------- W producer: one packed 128x128-code tile per k-block ----------------
            if (lane == 0) {
                Ring ring;
                TcPiece pc;
                TcWalk wk;
                wk.start(cluster);
                bool ok = true;
                while (ok && wk.next(sc, p, nclusters, pc)) {
                    const int nt = 2 * pc.ntp + (int)rank;
                    if (nt >= p.NT1) continue;                              // the second half of the last, odd pair
                    const ExpertDev& ex = p.ex[pc.e];
                    const uint32_t bytes = (uint32_t)ex.tile_stride;        // codes + the tile's scales / zero-points
                    const uint8_t* src = ex.tiles + ((size_t)nt * p.KB + pc.kb0) * bytes;
                    for (int kb = pc.kb0; kb < pc.kb1; ++kb, src += bytes) {
                        if (!(ok = mbar_wait(bar_wempty + 8 * ring.stage, ring.phase ^ 1u, s_abort, p.status))) break;
                        const uint32_t full = bar_wfull + 8 * ring.stage;
                        mbar_expect_tx(full, bytes);
                        bulk_load(sbase + L::w_off + ring.stage * p.wstage, src, bytes, full);
                        ring.advance(p.nw);
                    }
                }
            }
            __syncwarp();
            cluster_wait();
        } else if (warp == 1 && rank == 0) {
            // ---------------- MMA issuer (the leading CTA's, for the pair) ----------------
            // (Its waits spin on the plain try_wait: they sit on the critical path and coming round a short spin is
            // faster than waking from the hinted sleep.)
            // The WHOLE warp walks the pieces, so that control flow stays warp-uniform, and one elected lane issues
            // straight-line MMAs whose operands were all computed beforehand: issued from a loop that only lane 0
            // runs, every MMA costs ~250 cycles.
            TcPiece pc;
            TcWalk wk;
            wk.start(cluster);
            bool ok = true;
            uint32_t step = 0;
            int buf = 0;
            uint32_t buf_phase = 1;                        // parity of "empty" for the buffers of this round
            auto next_buf = [&]() { if (++buf == NACC) { buf = 0; buf_phase ^= 1u; } };
            while (ok && wk.next(sc, p, nclusters, pc)) {
                const int nh = NH == 1 ? 1 : (pc.rows > L::HC ? 2 : 1);
                const int group = p.ex[pc.e].group;
                // A per-channel expert's half tile h stays in buffer (buf + h) of the rotation for the whole piece.
                const bool keep = group == 0;
                const int steps = keep || group >= 128 ? 8 : group >> 4;         // MMAs into one accumulator buffer
                int kb0 = pc.kb0;
                const uint32_t idesc0 = umma_idesc_pair(half_cols<L::HC>(pc.rows, 0)), idesc1 = KS == 2 ? idesc0 : umma_idesc_pair(half_cols<L::HC>(pc.rows, nh - 1));
                // eight MMAs: one k-block (xd: its token rows, at: its weights) into the accumulator at d
                auto mma_kblock = [&](uint32_t d, uint32_t at, uint64_t xd, uint32_t idesc, uint32_t add = 0u) {
#pragma unroll
                    for (int i = 0; i < 8; ++i) umma_pair_ts(d, at + 8 * i, xd + (i >> 2) * (L::XR * 8) + (i & 3) * 2, idesc, i > 0 ? 1u : add);
                };
                // This warp's instructions are on the critical path of every step (the tensor core runs dry while it waits, votes
                // and commits), so the loops of the common formats hold as few of them as can be (8192 rows x 4096 x 4096, per
                // channel: 194 us, with one loop for every format 211).
                const uint32_t xd0 = sbase, at0 = tmem_base + L::a_base;
                if (keep) {
                    const int b1 = buf + 1 == NACC ? 0 : buf + 1;
                    const uint32_t ph1 = b1 == 0 ? buf_phase ^ 1u : buf_phase;
                    const uint32_t d0 = tmem_base + buf * L::HC, d1 = tmem_base + b1 * L::HC;
                    ok = warp_wait(bar_accempty + 8 * buf, buf_phase, s_abort, p.status);
                    if (nh == 2) ok &= warp_wait(bar_accempty + 8 * b1, ph1, s_abort, p.status);
                    ok = __all_sync(0xffffffffu, ok);
                    uint32_t add = 0u;
#pragma unroll 1
                    for (; ok && kb0 < pc.kb1; kb0 += KS, ++step) {
                        const uint32_t st = step % NX;
                        ok = warp_wait(bar_xfull + 8 * st, step / NX & 1u, s_abort, p.status);
                        ok &= warp_wait(bar_afull + 8 * (step % NA), step / NA & 1u, s_abort, p.status);
                        tc_fence_after();
                        const uint64_t xd = umma_desc_sw128(xd0 + st * L::xstage);
                        const uint32_t at = at0 + (step % NA) * (KS * TC_A_COLS);
                        const bool two = KS == 2 ? kb0 + 1 < pc.kb1 : nh == 2;
                        if (elect_one()) {
                            mma_kblock(d0, at, xd, idesc0, add);
                            if (two) {
                                if (KS == 2) mma_kblock(d0, at + TC_A_COLS, xd + L::xhalf / 16, idesc0, 1u);
                                else mma_kblock(d1, at, xd + L::xhalf / 16, idesc1, add);
                            }
                            umma_commit_pair(bar_done + 8 * st);
                        }
                        add = 1u;
                        ok = __all_sync(0xffffffffu, ok);
                    }
                    if (ok && elect_one()) {
                        umma_commit_pair(bar_accfull + 8 * buf);
                        if (nh == 2) umma_commit_pair(bar_accfull + 8 * (NACC + b1));
                    }
                    __syncwarp();
                    for (int h = 0; h < nh; ++h) next_buf();
                    continue;
                }
                if (steps == 8 && (KS == 2 || nh == 2)) {
                    // two buffers a step
#pragma unroll 1
                    for (; ok && kb0 + KS <= pc.kb1; kb0 += KS, ++step) {
                        const uint32_t st = step % NX;
                        const int b1 = buf + 1 == NACC ? 0 : buf + 1;
                        const uint32_t ph1 = b1 == 0 ? buf_phase ^ 1u : buf_phase;
                        ok = warp_wait(bar_xfull + 8 * st, step / NX & 1u, s_abort, p.status);
                        ok &= warp_wait(bar_afull + 8 * (step % NA), step / NA & 1u, s_abort, p.status);
                        ok &= warp_wait(bar_accempty + 8 * buf, buf_phase, s_abort, p.status);
                        if (KS == 2) ok &= warp_wait(bar_accempty + 8 * b1, ph1, s_abort, p.status);
                        tc_fence_after();
                        const uint64_t xd = umma_desc_sw128(xd0 + st * L::xstage);
                        const uint32_t at = at0 + (step % NA) * (KS * TC_A_COLS);
                        if (KS == 2) {
                            if (elect_one()) {
                                mma_kblock(tmem_base + buf * L::HC, at, xd, idesc0);
                                umma_commit_pair(bar_accfull + 8 * buf);
                                mma_kblock(tmem_base + b1 * L::HC, at + TC_A_COLS, xd + L::xhalf / 16, idesc0);
                                umma_commit_pair(bar_done + 8 * st);
                            }
                        } else {
                            if (elect_one()) {
                                mma_kblock(tmem_base + buf * L::HC, at, xd, idesc0);
                                umma_commit_pair(bar_accfull + 8 * buf);
                            }
                            __syncwarp();
                            ok &= warp_wait(bar_accempty + 8 * b1, ph1, s_abort, p.status);
                            tc_fence_after();
                            if (elect_one()) {
                                mma_kblock(tmem_base + b1 * L::HC, at, xd + L::xhalf / 16, idesc1);
                                umma_commit_pair(bar_done + 8 * st);
                            }
                        }
                        buf_phase = ph1;
                        buf = b1;
                        next_buf();
                        ok = __all_sync(0xffffffffu, ok);
                    }
                }
                if (KS == 1 && steps == 8 && nh == 1) {
                    // one buffer a step
#pragma unroll 1
                    for (; ok && kb0 < pc.kb1; ++kb0, ++step) {
                        const uint32_t st = step % NX;
                        ok = warp_wait(bar_xfull + 8 * st, step / NX & 1u, s_abort, p.status);
                        ok &= warp_wait(bar_afull + 8 * (step % NA), step / NA & 1u, s_abort, p.status);
                        ok &= warp_wait(bar_accempty + 8 * buf, buf_phase, s_abort, p.status);
                        tc_fence_after();
                        const uint64_t xd = umma_desc_sw128(xd0 + st * L::xstage);
                        if (elect_one()) {
                            mma_kblock(tmem_base + buf * L::HC, at0 + (step % NA) * (KS * TC_A_COLS), xd, idesc0);
                            umma_commit_pair(bar_done + 8 * st);
                        }
                        next_buf();
                        ok = __all_sync(0xffffffffu, ok);
                    }
                }
                // groups narrower than 128 k, and the odd k-block of a step of two
                for (; ok && kb0 < pc.kb1; kb0 += KS) {
                    const int nk = min(KS, pc.kb1 - kb0);
                    ok = warp_wait(bar_xfull + 8 * (step % NX), step / NX & 1u, s_abort, p.status);
                    ok &= warp_wait(bar_afull + 8 * (step % NA), step / NA & 1u, s_abort, p.status);
                    tc_fence_after();
                    const uint32_t done = bar_done + 8 * (step % NX);
                    const uint64_t xdesc = umma_desc_sw128(sbase + (step % NX) * L::xstage);
                    // sub-steps: the half tiles of the k-block, or the k-blocks of the step.  Sub-step u is drained by epilogue
                    // group u (see there), so they take turns group by group and both epilogue groups always have a buffer.
                    const int nu = KS == 2 ? nk : nh;
#pragma unroll 1
                    for (int i0 = 0; i0 < 8; i0 += steps) {
#pragma unroll 1
                        for (int u = 0; u < nu; ++u) {
                            const int h = KS == 2 ? 0 : u, kk = KS == 2 ? u : 0;
                            const uint32_t a_tmem = tmem_base + L::a_base + ((step % NA) * KS + kk) * TC_A_COLS + 8 * i0;
                            const uint32_t idesc = h ? idesc1 : idesc0;
                            const uint64_t bd = xdesc + u * (L::xhalf / 16) + (i0 >> 2) * (L::XR * 8) + (i0 & 3) * 2;
                            const uint32_t d = tmem_base + buf * L::HC;
                            const uint32_t full = u + 1 == nu && i0 + steps == 8 ? done : bar_accfull + 8 * (u * NACC + buf);
                            ok &= warp_wait(bar_accempty + 8 * buf, buf_phase, s_abort, p.status);
                            tc_fence_after();
                            if (elect_one()) {
                                if (steps == 8) {
                                    mma_kblock(d, a_tmem, bd, idesc);
                                } else {
                                    umma_pair_ts(d, a_tmem, bd, idesc, 0u);
                                    umma_pair_ts(d, a_tmem + 8, bd + 2, idesc, 1u);
                                    if (steps == 4) {
                                        umma_pair_ts(d, a_tmem + 16, bd + 4, idesc, 1u);
                                        umma_pair_ts(d, a_tmem + 24, bd + 6, idesc, 1u);
                                    }
                                }
                                umma_commit_pair(full);
                            }
                            __syncwarp();
                            next_buf();
                        }
                    }
                    ok = __all_sync(0xffffffffu, ok);
                    ++step;
                }
            }
        }
    } else if (warp < L::epi_warp0) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(L::regs_dq));
        // ---------------- dequant warps: thread = channel = TMEM lane ----------------
        TcDequant d;
        d.bar_wfull = bar_wfull; d.bar_wempty = bar_wempty; d.bar_done = bar_done;
        d.afull0 = mapa(bar_afull, 0);
        d.row = (warp & 3) * 32 + lane;
        d.lane_tmem = tmem_base + ((uint32_t)((warp & 3) * 32) << 16) + L::a_base;
        d.nw = p.nw; d.wstage = p.wstage;
        d.my_group = (uint32_t)((warp - 4) >> 2);
        d.step = 0;
        const unsigned char* wtiles = smem + L::w_off;
        TcPiece pc;
        TcWalk wk;
        wk.start(cluster);
        bool ok = true;
        while (ok && wk.next(sc, p, nclusters, pc)) {
            const ExpertDev& ex = p.ex[pc.e];
            const int nt = 2 * pc.ntp + (int)rank, nkb = pc.kb1 - pc.kb0;
            if (nt >= p.NT1) { ok = dequant_none<TN>(d, sh, nkb, p.status); continue; }
            const bool has_zeros = ex.has_zeros != 0, tile_zeros = has_zeros && ex.group != 0;
            const int per = moqe_groups_per_tile(ex.group);
            float z = (float)(1 << (ex.bits - 1));
            if (has_zeros && ex.group == 0) z = __bfloat162float(ex.zeros_pc[nt * 128 + d.row]);
            const uint32_t zpc = neg_z(z);
            switch (ex.bits) {
                case 4: ok = dequant_piece<TN, 4>(d, sh, wtiles, nkb, per, zpc, tile_zeros, p.status); break;
                case 8: ok = dequant_piece<TN, 8>(d, sh, wtiles, nkb, per, zpc, tile_zeros, p.status); break;
                case 3: ok = dequant_piece<TN, 3>(d, sh, wtiles, nkb, per, zpc, tile_zeros, p.status); break;
                default: ok = dequant_piece<TN, 2>(d, sh, wtiles, nkb, per, zpc, tile_zeros, p.status); break;
            }
        }
    } else {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(L::regs_epi));
        // ---------------- epilogue warps: scale-and-accumulate, then store ----------------
        // Two groups of four warps.  Of a tile with two half tiles each group drains one, of a step with two k-blocks each
        // drains one (an accumulator buffer then costs a warp one wait for all its columns); otherwise both drain every
        // buffer, half the columns each.
        // (Each of the two sub-steps has its own accfull barriers: a wait tells only two phases of a barrier apart, so a barrier
        // is waited on by the warps that its buffer's reuse waits for, and by nobody who could fall two uses behind.)
        const int ew = warp - L::epi_warp0, quarter = warp & 3, eg = ew >> 2;
        const int row = quarter * 32 + lane;               // channel inside the 128-channel tile = TMEM lane
        const uint32_t accempty0 = mapa(bar_accempty, 0);
        const uint32_t lane_tmem = tmem_base + ((uint32_t)(quarter * 32) << 16);
        const uint32_t saved = smem_u32(sh.walk[ew]);
        int* my_perm = sh.perm[ew];                        // private to this warp: no cross-warp barrier
        TcPiece pc;
        TcWalk wk;
        wk.start(cluster);
        bool ok = true;
        int buf = 0;
        uint32_t full_phase = 0;                           // bit i: parity of the next arrival on accfull[i]
        uint32_t step = 0, xphase = 0;                     // steps so far; parity of the exchange
        while (ok && wk.next(sc, p, nclusters, pc)) {
            const ExpertDev& ex = p.ex[pc.e];
            int nt = 2 * pc.ntp + (int)rank, n = nt * 128 + row;
            bool active = nt < p.NT1;
            const int nh = NH == 1 ? 1 : (pc.rows > L::HC ? 2 : 1);
            // the columns this warp stores: ncol (may be <= 0) from token tok0 of the tile on
            const int hs = nh == 2 ? half_split<L::HC>(pc.rows) : L::HC / 2;
            int tok0 = eg * hs, ncol = min(hs, pc.rows - tok0);
            __syncwarp();
#pragma unroll
            for (int i = 0; i < L::EC / 32; ++i) {
                const int col = i * 32 + lane;
                my_perm[col] = col < ncol ? __ldcg(p.perm + pc.m0 + tok0 + col) : -1;
            }
            // What only the end of the piece asks for waits in shared memory: the drain loops have no registers for it, and the copies that
            // the compiler spilled instead were loaded again inside them.
            sts_v4(saved, pc.e, pc.ntp, pc.rows, pc.tile);
            sts_v4(saved + 16, pc.kb0, pc.kb1, wk.t, wk.e);
            sts_v4(saved + 32, wk.u, wk.ue, 0, 0);
            __syncwarp();
            float acc[L::DC];
#pragma unroll
            for (int i = 0; i < L::DC; ++i) acc[i] = 0.f;
            const bool keep = ex.group == 0;
            const int per = moqe_groups_per_tile(ex.group), nkb = pc.kb1 - pc.kb0;
            const float s_pc = keep && active ? __half2float(ex.scales_pc[n]) * W8_PRESCALE : 0.f;   // (weights are unpacked as (c - z) * 2^-13)
            const bool alone = KS == 2 || nh == 2;             // a buffer is drained by one group
            const uint32_t freed = alone ? 2u : 1u;
            const int col0 = alone ? 0 : tok0;                 // first column drained, and how many hold a token
            const int dcol = KS == 2 ? pc.rows : ncol;
            if (keep) {
                // Per channel: a half tile's buffer is drained once.  (Apart from the groups' loops, whose scales and counts are then not
                // alive here: 28224 rows of 256 -> 1024 channels 34.6 us; 40.7 where both share one drain, and a piece of two k-blocks
                // pays for its spills.)
                const int nu = KS == 2 ? 1 : nh;
#pragma unroll 1
                for (int u = 0; u < nu; ++u) {
                    const int fb = u * NACC + buf;
                    if (!alone || u == eg) {
                        ok &= warp_wait(bar_accfull + 8 * fb, (full_phase >> fb) & 1u, s_abort, p.status);
                        tc_fence_after();
#pragma unroll
                        for (int c = 0; c < L::DC / 32; ++c)
                            if (32 * c < dcol) {
                                uint32_t v[32];
                                tmem_ld32(lane_tmem + buf * L::HC + col0 + 32 * c, v);
                                tmem_ld_wait();
                                fma_cols32(acc + 32 * c, v, s_pc);
                            }
                        tc_fence_before();
                        __syncwarp();
                        remote_arrive_if(lane == 0, accempty0 + 8 * buf, freed);
                    }
                    full_phase ^= 1u << fb;
                    if (++buf == NACC) buf = 0;
                }
                step += (nkb + KS - 1) / KS;
                ok = __all_sync(0xffffffffu, ok);
            } else {
                // Scales come straight from the tiles in global memory (the packed tile has just been fetched, so they are in L2),
                // two drains ahead of their use.  Handed on by the dequant warps through shared memory and a barrier of their own,
                // they cost both roles some 200 cycles a k-block.
                const int mg = ex.has_zeros ? 512 : 256, round = KS * ex.tile_stride;
                const unsigned char* meta = ex.tiles + ((size_t)(active ? nt : 0) * p.KB + pc.kb0) * ex.tile_stride + moqe_tile_bytes(ex.bits) + row * 2;
                const int off_end = (nkb - 1) * ex.tile_stride + (per - 1) * mg;
                int off = min(KS == 2 ? eg * ex.tile_stride : 0, (nkb - 1) * ex.tile_stride), oj = 0;
                auto fetch_scale = [&]() { return __ldg(reinterpret_cast<const unsigned short*>(meta + off)); };
                auto next_scale = [&](bool one) {                      // one: a group to a k-block
                    if (one) off = min(off + round, off_end);
                    else {
                        const bool wrap = ++oj == per;
                        off = min(off + (wrap ? round - (per - 1) * mg : mg), off_end);
                        oj = wrap ? 0 : oj;
                    }
                };
                unsigned short s_now = fetch_scale();                  // (as loaded: converting waits for the load)
                next_scale(per == 1);
                unsigned short s_next = fetch_scale();
                // waits for an accumulator buffer, adds it to the sums and hands it back
                auto drain = [&](auto chunks, bool one, uint32_t bar, uint32_t phase, int b) {
                    ok &= warp_wait(bar, phase, s_abort, p.status);
                    tc_fence_after();
                    const uint32_t src = lane_tmem + b * L::HC + col0;
                    float sv = 0.f;
#pragma unroll
                    for (int c = 0; c < L::DC / 32; ++c) {
                        if (decltype(chunks)::value > 0 ? c < decltype(chunks)::value : 32 * c < dcol) {
                            uint32_t v[32];
                            tmem_ld32(src + 32 * c, v);
                            if (c == 0) {
                                // (while the load is under way)
                                sv = __half2float(__ushort_as_half(s_now)) * W8_PRESCALE;
                                s_now = s_next;
                                next_scale(one);
                                s_next = fetch_scale();
                            }
                            tmem_ld_wait();
                            fma_cols32(acc + 32 * c, v, sv);
                        }
                    }
                    tc_fence_before();
                    __syncwarp();
                    remote_arrive_if(lane == 0, accempty0 + 8 * b, freed);
                };
                int left = nkb;
                // The loop is kept short, since a warp gets an instruction through every nine cycles or so and nothing else of
                // the epilogue runs in parallel.
                const bool by_done = !alone || eg == 1;            // announced by the step's own barrier if it is the last group
                const int mine = alone ? eg : 0, uses = alone ? 2 : 1;
                auto steps = [&](auto chunks, auto one) {
                    constexpr bool ONE = decltype(one)::value;     // a group to a k-block (the common formats)
#pragma unroll 1
                    for (; ok && left >= KS; left -= KS) {
#pragma unroll 1
                        for (int g = 1; ; ++g) {
                            const bool last = ONE || g == per;
                            int ob = buf + mine;
                            if (ob >= NACC) ob -= NACC;
                            const bool dn = by_done && last;
                            const int fb = ONE ? ob : (mine ? NACC : 0) + ob;
                            drain(chunks, ONE, dn ? bar_done + 8 * (step % NX) : bar_accfull + 8 * fb, dn ? step / NX & 1u : (full_phase >> fb) & 1u, ob);
                            if (alone) {
                                full_phase ^= 1u << buf;
                                if (!ONE && !last) full_phase ^= 1u << (NACC + (buf + 1 == NACC ? 0 : buf + 1));
                            } else if (!last) {
                                full_phase ^= 1u << buf;
                            }
                            buf += uses;
                            if (buf >= NACC) buf -= NACC;
                            if (last) break;
                        }
                        ++step;
                        ok = __all_sync(0xffffffffu, ok);
                    }
                };
                auto run = [&](auto one) {
                    // The number of 32-column chunks is fixed at compile time: no branch between them, and the loads of a chunk start before
                    // the sums of the last are done.  128 tokens, two chunks, 18944 x 3584 in 4-bit g64 and g32: 32.6 and 51.3 us, with
                    // the branches 36.4 and 58.2; a single chunk of narrow groups (50.8 against 57.4 in g32) and the smallest tile
                    // (96 rows x 4096 x 11008: 38.3 against 39.0) are better with them.
                    constexpr bool ONE = decltype(one)::value;
                    if constexpr (TN == 64) {
                        steps(std::integral_constant<int, 0>{}, one);
                    } else if constexpr (TN == 128) {
                        if (dcol > 32) steps(std::integral_constant<int, 2>{}, one);
                        else steps(std::integral_constant<int, ONE ? 1 : 0>{}, one);
                    } else {
                        const int nch = (dcol + 31) >> 5;
                        if (nch <= 1) steps(std::integral_constant<int, 1>{}, one);
                        else if (nch == 2) steps(std::integral_constant<int, 2>{}, one);
                        else if (nch == 3) steps(std::integral_constant<int, 3>{}, one);
                        else steps(std::integral_constant<int, 4>{}, one);
                    }
                };
                if (per == 1) run(std::true_type{});
                else run(std::false_type{});
                if constexpr (KS == 2) {
                    // The odd k-block of a piece: every group's buffer is drained, the last one being announced by the step's own barrier.
                    // (The loop is kept rolled: the kernel is fetched as it runs.)
                    if (ok && left > 0) {
#pragma unroll 1
                        for (int t = 0; t < per; ++t) {
                            const bool by_done = t + 1 == per;
                            if (eg == 0)
                                drain(std::integral_constant<int, 0>{}, false, by_done ? bar_done + 8 * (step % NX) : bar_accfull + 8 * buf, by_done ? step / NX & 1u : (full_phase >> buf) & 1u, buf);
                            if (!by_done) full_phase ^= 1u << buf;
                            if (++buf == NACC) buf = 0;
                        }
                        ++step;
                        ok = __all_sync(0xffffffffu, ok);
                    }
                }
            }
            if constexpr (KS == 2) {
                // the two groups hold sums over different k-blocks: each takes half of the columns and hands over the others
                float* x = reinterpret_cast<float*>(smem + L::xchg_off) + lane;
                float* out = x + ew * 1024;
                const float* in = x + (ew ^ 4) * 1024;
                // (on mbarriers: every wait of this kernel is bounded)
                const uint32_t xfull = bar_xchg, xempty = bar_xchg + 8 * TC_EPI;
                ok &= warp_wait(xempty + 8 * ew, xphase ^ 1u, s_abort, p.status);
#pragma unroll
                for (int i = 0; i < 32; ++i) out[i * 32] = eg ? acc[i] : acc[i + 32];
                __syncwarp();
                mbar_arrive_if(lane == 0, xfull + 8 * ew);
                ok &= warp_wait(xfull + 8 * (ew ^ 4), xphase, s_abort, p.status);
#pragma unroll
                for (int i = 0; i < 32; ++i) acc[i] = (eg ? acc[i + 32] : acc[i]) + in[i * 32];
                __syncwarp();
                mbar_arrive_if(lane == 0, xempty + 8 * (ew ^ 4));   // (plain stores follow, which its release orders behind the reads)
                xphase ^= 1u;
                ok = __all_sync(0xffffffffu, ok);
            }
            {
                int unused;
                lds_v4(saved, pc.e, pc.ntp, pc.rows, pc.tile);
                lds_v4(saved + 16, pc.kb0, pc.kb1, wk.t, wk.e);
                lds_v4(saved + 32, wk.u, wk.ue, unused, unused);
                nt = 2 * pc.ntp + (int)rank; n = nt * 128 + row;
                active = nt < p.NT1;
                const int h0 = NH > 1 && pc.rows > L::HC ? half_split<L::HC>(pc.rows) : L::HC / 2;
                tok0 = eg * h0; ncol = min(h0, pc.rows - tok0);
            }
            if (!ok) break;
            if (!active) continue;
            if (pc.kb0 != 0 || pc.kb1 != p.KB) {
                // part of a tile: park this warp's sums, announce, and add everything up if this was the last arrival
                const int C = sc.C, Gs = sc.Gs, first = sc.base[pc.e] + (pc.tile * p.KB - sc.us[pc.e]) * sc.w[pc.e];
                const int c_a = first * Gs / C, c_b = (first + (p.KB - 1) * sc.w[pc.e]) * Gs / C;
                const size_t slot = (size_t)p.cols * 128;
                auto slot_of = [&](int c, int which) { return p.partials + ((size_t)(c * 2 + which) * 2 + rank) * slot + (size_t)tok0 * 128 + row * 4; };
                unsigned* counter = p.counters + (c_a * 2 + (int)rank) * TC_EPI + ew;
                const unsigned others = (unsigned)(c_b - c_a);
                // A tile's first part is the last thing its cluster does, so the others' sums are usually there already: then this
                // warp's own stay in registers (parking them takes 2.5 us).
                unsigned arrived = 0;
                if (pc.kb0 == 0) {
                    if (lane == 0) arrived = ld_acquire_gpu(counter);
                    arrived = __shfl_sync(0xffffffffu, arrived, 0);
                }
                const bool direct = arrived == others;
                if (!direct) {
                    float* dst = slot_of(cluster, pc.kb0 == 0 ? 1 : 0);
#pragma unroll
                    for (int i = 0; i < L::EC; i += 4)
                        if (i < ncol) __stcg(reinterpret_cast<float4*>(dst + i * 128), make_float4(acc[i], acc[i + 1], acc[i + 2], acc[i + 3]));
                    __syncwarp();
                    // one acquire-release increment: the release side publishes the warp's parked sums (ordered before it by the
                    // warp barrier above), the acquire side lets the last arriver read everybody else's
                    if (lane == 0) asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], 1;" : "=r"(arrived) : "l"(counter) : "memory");
                    arrived = __shfl_sync(0xffffffffu, arrived, 0);
                    if (arrived != others) continue;
#pragma unroll
                    for (int i = 0; i < L::EC; ++i) acc[i] = 0.f;
                }
                __syncwarp();
                // added in cluster order (whoever arrives last: the first cluster's sums are the ones that may be in registers)
                constexpr int CB = TN == 64 ? 2 : 1, CC = 32;
#pragma unroll 1
                for (int c = c_a + (direct ? 1 : 0); c <= c_b; c += CB) {
#pragma unroll
                    for (int i0 = 0; i0 < L::EC; i0 += CC)
                        if (i0 < ncol) {
                            float4 v[CB][CC / 4];
#pragma unroll
                            for (int b = 0; b < CB; ++b) {
                                const float* src = slot_of(min(c + b, c_b), c + b == c_a ? 1 : 0) + i0 * 128;
#pragma unroll
                                for (int i = 0; i < CC / 4; ++i)
                                    v[b][i] = i0 + 4 * i < ncol && c + b <= c_b ? __ldcg(reinterpret_cast<const float4*>(src + i * 512)) : make_float4(0.f, 0.f, 0.f, 0.f);
                            }
#pragma unroll
                            for (int b = 0; b < CB; ++b)
#pragma unroll
                                for (int i = 0; i < CC / 4; ++i) {
                                    acc[i0 + 4 * i] += v[b][i].x;
                                    acc[i0 + 4 * i + 1] += v[b][i].y;
                                    acc[i0 + 4 * i + 2] += v[b][i].z;
                                    acc[i0 + 4 * i + 3] += v[b][i].w;
                                }
                        }
                }
                if (lane == 0) *counter = 0u;
            }
            // Store: lanes hold neighbouring channels, registers tokens.  Four neighbouring lanes transpose four tokens between
            // them (two exchanges), so that a lane writes four channels of one token.  The store is predicated, not branched
            // around: with a branch each, 64 stores took a warp 9500 cycles.
            const int sub = lane & 3;
            uint16_t* y = p.Y + (n & ~3);
            const int* to_list = my_perm + sub;
            const bool in_n = n < p.N;
#pragma unroll
            for (int i0 = 0; i0 < L::EC; i0 += 16)
                if (i0 < ncol) {
#pragma unroll
                    for (int i = i0; i < i0 + 16; i += 4) {
                        const uint32_t p01 = pack_bf16x2(acc[i], acc[i + 1]), p23 = pack_bf16x2(acc[i + 2], acc[i + 3]);
                        const uint32_t q01 = __shfl_xor_sync(0xffffffffu, p01, 1), q23 = __shfl_xor_sync(0xffffffffu, p23, 1);
                        const uint32_t a = __byte_perm(p01, q01, sub & 1 ? 0x3276u : 0x5410u);       // two channels of token i + (sub & 1)
                        const uint32_t b = __byte_perm(p23, q23, sub & 1 ? 0x3276u : 0x5410u);       // ... of token i + 2 + (sub & 1)
                        const uint32_t other = __shfl_xor_sync(0xffffffffu, sub & 2 ? a : b, 2);
                        const int to = to_list[i];
                        uint16_t* at = y + (size_t)(uint32_t)max(to, 0) * (uint32_t)p.N;
                        asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.b32 q, %3, 0;\n\t@q st.global.v2.b32 [%0], {%1, %2};\n\t}"
                                     ::"l"(at), "r"(sub & 2 ? other : a), "r"(sub & 2 ? b : other), "r"((int)(in_n && to >= 0)) : "memory");
                    }
                }
        }
    }

    // ---------------- teardown ----------------
    tc_fence_before();
    __syncthreads();
    if (*s_abort) {
        // let bulk copies that may still be in flight land before the shared memory is released
        unsigned long long t0 = global_ns();
        while (global_ns() - t0 < 200000ull) __nanosleep(1000);
    }
    cluster_arrive();
    cluster_wait();                                        // the peer no longer touches this CTA's barriers or TMEM
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc_pair(tmem_base, 512);
    }
}

// columns of a parked partial sum: no tile has more tokens than the batch
int tc_cols(int M) { return M >= 256 ? 256 : (M + 31) / 32 * 32; }

}  // namespace

size_t tc_zero_bytes() { return (size_t)TC_MAX_CLUSTERS * 2 * TC_EPI * sizeof(uint32_t); }

size_t tc_workspace_bytes(int M, int K, int E, int Np) {
    (void)K; (void)E; (void)Np;
    return (size_t)TC_MAX_CLUSTERS * 4 * tc_cols(M) * 128 * sizeof(float);
}

moqe_status launch_qgemm_tc(const void* X, int M, int N, int K, const moqe_expert* const* ex, int E, void* Y,
                            const int32_t* perm, const int32_t* offsets, uint32_t* counters, void* ws, size_t ws_bytes, int tile_tokens,
                            cudaStream_t st) {
    if (M == 0) return MOQE_OK;
    if (!ws || ws_bytes < tc_workspace_bytes(M, K, E, ex[0]->Np)) return MOQE_ERR_WORKSPACE;
    EncodeTiledFn enc = encode_tiled_fn();
    if (!enc) return MOQE_ERR_CUDA;
    // Tile by batch size (the routing is not known here): LLaMA blocks, three experts, rows dealt evenly, 64 / 128 / 256
    // tokens: 192 rows 235 / 275 / 302 us, 256 rows 367 / 299 / 318, 384 rows 383 / 323 / 346, 512 rows 474 / 489 / 414.
    // A layer that would leave clusters without a tile takes smaller ones while they still fit one round (980 rows of
    // 256 x 1024, 128 against 256 tokens: 11 / 16 us).
    const int sms = device_sm_count();
    const int clusters = sms / 2 < TC_MAX_CLUSTERS ? sms / 2 : TC_MAX_CLUSTERS;
    int tile = tile_tokens ? tile_tokens : (M > 448 ? 256 : (M > 192 ? 128 : 64));
    const int ntp = (ex[0]->Np / 128 + 1) / 2;
    if (!tile_tokens)
        while (tile > 64 && (long long)(2 * M / tile + E) * ntp <= clusters) tile /= 2;
    // tensor map over X[M][K] bf16: boxes of 64 k x XR rows, 128-byte swizzle, zero fill outside
    CUtensorMap tmap;
    cuuint64_t gdim[2] = {(cuuint64_t)K, (cuuint64_t)M};
    cuuint64_t gstride[1] = {(cuuint64_t)K * 2};
    cuuint32_t box[2] = {64, tile == 64 ? 32u : 64u}, estr[2] = {1, 1};
    if (enc(&tmap, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(X), gdim, gstride, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
            CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
        return MOQE_ERR_CUDA;
    TcParams p;
    int stride = 0;
    for (int e = 0; e < E; ++e) {
        p.ex[e] = ex[e]->dev();
        stride = p.ex[e].tile_stride > stride ? p.ex[e].tile_stride : stride;
    }
    p.perm = perm; p.offsets = offsets; p.X = (const uint16_t*)X; p.Y = (uint16_t*)Y; p.status = device_status_word();
    p.counters = counters;
    p.partials = (float*)ws;
    p.M = M; p.N = N; p.K = K; p.KB = ex[0]->Kp / 128; p.E = E; p.NT1 = ex[0]->Np / 128; p.NTP = (p.NT1 + 1) / 2;
    p.cols = tc_cols(M);
    p.split = tile_tokens == 0 && tc_split_fits(clusters, p.KB) ? 1 : 0;
    auto launch = [&](auto kernel, int threads, int smem, int w_bytes, std::atomic<unsigned long long>& attr) -> bool {
        p.wstage = (stride + 127) / 128 * 128;
        p.nw = w_bytes / p.wstage < TC_NW_MAX ? w_bytes / p.wstage : TC_NW_MAX;
        if (!ensure_dynamic_smem((const void*)kernel, smem, attr)) return false;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(2 * clusters); cfg.blockDim = dim3(threads); cfg.dynamicSmemBytes = smem; cfg.stream = st;
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        at[0].val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = at; cfg.numAttrs = 1;
        return cudaLaunchKernelEx(&cfg, kernel, p, tmap) == cudaSuccess;
    };
    auto run = [&](auto tag) {
        using L = TcCfg<decltype(tag)::value>;
        static std::atomic<unsigned long long> attr{0};
        return launch(qgemm_tc_kernel<decltype(tag)::value>, L::threads, L::dyn_bytes, L::w_bytes, attr);
    };
    const bool launched = tile == 256 ? run(std::integral_constant<int, 256>{})
                                      : (tile == 128 ? run(std::integral_constant<int, 128>{}) : run(std::integral_constant<int, 64>{}));
    if (!launched) { cudaGetLastError(); return MOQE_ERR_CUDA; }
    count_launch();
    return cuda_ok(cudaGetLastError());
}

}  // namespace moqe
