// The two passes of the wide-row path (see harp_split.cu) fed by the copy engine.
//
// The mma.sync passes of harp_split.cu spend 60 % of a tile's time on moving it: cp.async in and 16-byte stores out hold the
// issuing warps at the rate at which the load/store unit takes 32-byte runs (d = 14336, upper pass: 14.8 k cycles a tile with
// three CTAs on an SM, 5 k of them products).  Bulk tensor copies move the same boxes without a warp: runs of 32 bytes in 1.4
// cycles each one way and 3.3 both ways (4.6 to 4.9 TB/s), of 64 bytes and more at 5.5 to 6 TB/s.  So teams of warps multiply
// tiles in place while other buffers of theirs are stored and refilled; all teams share the fragments of the CTA's column group.
//
//   d = 14336, 32768 rows: 888 -> 740 us;  d = 28672, 16384 rows: 1070 -> 750 us;  d = 8192, 16384 rows: 318 -> 212 us;
//   d = 11008, 16384 rows: 384 -> 270 us (dense upper blocks);  d = 5120, 16384 rows: 221 -> 136 us;
//   d = 8192, 64 rows: 12.9 -> 8.0 us;  d = 11008, 1 row: 9.3 -> 7.3 us.
// With the products left out the upper passes take 95 to 100 % of their time and the slab pass 80 %: the copies bound them.
// (One product with 64 x 64 blocks instead of a slab's first two phases was as fast, but rounds once where the other kernels
// round twice; results now are the same bits whichever kernel takes a batch.)
//
// The tile's layout is what the copy engine writes, chosen so that the 16-byte accesses of a quarter-warp (two rows, four
// local indices) hit eight bank groups:
//   slab pass   [box of 64 coordinates][row][128 bytes], 128-byte swizzle, boxes 128 bytes apart beyond their size: an index
//               step of one chunk or one box moves the swizzle by one, lanes hold the local indices 2q, 2q+1;
//   upper pass  [half of the rows][row][outer digit][inner digit][column of 32 or 64 bytes], 32- or 64-byte swizzle.  The inner digit's
//               radix is odd (or there is one digit), so a step of either digit is an odd number of columns; the two rows of a
//               quarter-warp come from the two halves, whose distance moves the top bit of the swizzle by one.
// Columns of 64 bytes double the fragments of a column group and halve the number of groups.  One phase of sixteen takes them (d = 8192,
// 16384 rows: 223 -> 218 us; 16 groups instead of 32 also fill 144 SMs instead of 128), and so do two phases of eight for
// batches that fill the SMs, with the fragments in registers so that three buffers fit (d = 14336, 32768 rows: 750 -> 667 us;
// d = 28672, 4096 rows: 190 -> 175 us; with the fragments in shared memory and one buffer per team it was slower than columns of 32).
// So does one phase of eight (d = 4096, radix 8, 16384 rows: 119 -> 111 us).
// A slab's first two phases stay with one warp (its box, fragments in registers, no barrier between them).
#include <algorithm>
#include <new>
#include <vector>

#include "harp_fuse.h"
#include "harp_internal.h"
#include "harp_mma.cuh"
#include "harp_ring.h"
#include "harp_tm_ptx.cuh"

namespace {

using namespace harp_fuse;
using harp_tm::mbar_expect_tx;
using harp_tm::mbar_init;
using harp_tm::mbar_try;

constexpr int kMaxPipePhases = 3, kMaxPipeBufs = 4;
constexpr uint32_t kPipeSpin = 1u << 22;      // limit of every wait for a bulk copy

struct PipePhase {
    int32_t mode;              // 0 = the pair of phases inside a box; 1 = strided blocks, eight per item
    int32_t B, B_real;
    int32_t n_items, items_off;
    int32_t bfrag_off;         // word offset of the phase's fragments inside a column group's block
    int32_t lm;                // local index of slot j of lane q: lm * q + jr[j]
    int32_t jr[4];
    int32_t step[2];           // byte offset of local index r: (r * unit >> shift) * step[1] + (r * unit & mask) * step[0]
    int32_t unit, shift;
};

struct PipePass {
    int32_t n_phases, n_cg, MT, mt_shift;
    int32_t n_box, box_bytes, box_pitch;      // bulk copies of a tile, their size, their distance in shared memory
    int32_t row_bytes;                        // upper: distance of neighbouring rows of a half
    int32_t tile_bytes, n_buf;                // distance of a team's buffers, their number
    int32_t n_tiles, n_parts;                 // n_parts > 0: a CTA keeps its column group and takes every n_parts-th tile; 0: equal shares of the list
    const int32_t *tables;                    // byte offsets of the items
    int32_t tables_len;
    const uint32_t *bfrag;                    // fragments, frag_stride words per column group (the plan's copy, see harp_split.cu)
    int32_t frag_stride, smem_off, bfrag_words;   // part of them that the phases read from shared memory
    int32_t pair_off[2], pair_bwd;            // lower: fragments of the first two phases; octets first (transpose)
    PipePhase ph[kMaxPipePhases];
};

__device__ __forceinline__ uint32_t lds32p(uint32_t addr) {
    uint32_t v;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(addr));
    return v;
}
__device__ __forceinline__ void tma_load_4d(uint32_t dst, const CUtensorMap *map, int a, int b, int c, int d, uint32_t bar) {
    asm volatile("cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], [%6];"
                 ::"r"(dst), "l"(map), "r"(a), "r"(b), "r"(c), "r"(d), "r"(bar) : "memory");
}
__device__ __forceinline__ void tma_store_4d(const CUtensorMap *map, int a, int b, int c, int d, uint32_t src) {
    asm volatile("cp.async.bulk.tensor.4d.global.shared::cta.tile.bulk_group [%0, {%1, %2, %3, %4}], [%5];"
                 ::"l"(map), "r"(a), "r"(b), "r"(c), "r"(d), "r"(src) : "memory");
}

__device__ __forceinline__ uint32_t local_off(const PipePhase &ph, int r) {
    const int e = r * ph.unit;
    return (uint32_t)((e >> ph.shift) * ph.step[1] + (e & ((1 << ph.shift) - 1)) * ph.step[0]);
}

// The kinds of pass.  A team is a few warps with n_buf tile buffers of their own; tiles of the CTA's column group go to its
// teams in turn and a team's thread 0 issues its bulk copies.
//   lower8, upper8, upper8One   three teams of eight warps, at most 85 registers; lower8: a warp per box of 64 coordinates in the first two phases
//                    (upper8One: one phase, columns of 64 bytes)
//   upper8Wide       one team of sixteen warps, two phases, a warp's two octets of each with their fragments in registers
//   upper16          one phase of sixteen-wide blocks, 128 registers: two teams of eight warps
//   dense32, dense48 all upper stages as one block of up to 32 or 48: a warp holds sixteen rows of eight positions, the two
//                    octets of a tile make a team of two warps; three teams
enum Kind { kLower8, kUpper8, kUpper8One, kUpper8Wide, kUpper16, kDense32, kDense48 };
constexpr bool is_wide(int K) { return K == kUpper8One || K == kUpper8Wide || K == kUpper16; }
template <int K> struct KindOf {
    static constexpr bool lower = K == kLower8, b16 = K == kUpper16, wide = is_wide(K);
    static constexpr int ks = K == kDense32 ? 2 : K == kDense48 ? 3 : 0;
    static constexpr int team_warps = ks ? 2 : K == kUpper8Wide ? 16 : 8, team_threads = 32 * team_warps, teams = K == kUpper8Wide ? 1 : b16 ? 2 : 3, threads = teams * team_threads;
    static constexpr int swizzle_bits = lower ? 7 : wide ? 3 : 1;
};
template <int K> __device__ __forceinline__ uint32_t swz(uint32_t a) { return a ^ (((a >> 7) & (uint32_t)KindOf<K>::swizzle_bits) << 4); }

// Eight positions of sixteen rows through one dense block each (U <= 16 KS).  raw: slot s of this lane is coordinate
// 16 (s / 4) + q + 4 (s % 4); results replace the operands word by word.
// Fragments: [pair of positions][pair of column tiles][position of the pair][KS][lane][4 words].
template <int K, typename Mid>
__device__ __forceinline__ void dense_octet(uint32_t a0, uint32_t row8_off, int q, int U, uint32_t bfa, const Mid &mid) {
    constexpr int KS = KindOf<K>::ks;
    uint4 raw[4 * KS][2];
#pragma unroll
    for (int s = 0; s < 4 * KS; ++s) {
        const int u = 16 * (s / 4) + q + 4 * (s % 4);
        const uint32_t o = a0 + 32u * (uint32_t)u;
        raw[s][0] = u < U ? lds128(swz<K>(o)) : make_uint4(0u, 0u, 0u, 0u);
        raw[s][1] = u < U ? lds128(swz<K>(o + row8_off)) : make_uint4(0u, 0u, 0u, 0u);
    }
#pragma unroll
    for (int w = 0; w < 4; ++w) {
        uint32_t a[2][KS][4];
#pragma unroll
        for (int ks = 0; ks < KS; ++ks)
#pragma unroll
            for (int m = 0; m < 4; ++m) {
                const uint32_t x = word_of(raw[4 * ks + 2 * (m >> 1)][m & 1], w), y = word_of(raw[4 * ks + 2 * (m >> 1) + 1][m & 1], w);
                a[0][ks][m] = pair_lo(x, y);
                a[1][ks][m] = pair_hi(x, y);
            }
#pragma unroll
        for (int c = 0; c < KS; ++c) {
            uint4 f[2][KS];
#pragma unroll
            for (int ee = 0; ee < 2; ++ee)
#pragma unroll
                for (int t = 0; t < KS; ++t) f[ee][t] = lds128(bfa + 512u * (uint32_t)(((w * KS + c) * 2 + ee) * KS + t));
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                float acc[2][4];
#pragma unroll
                for (int ee = 0; ee < 2; ++ee)
#pragma unroll
                    for (int ks = 0; ks < KS; ++ks) {
                        const int at = 2 * (k * KS + ks);
                        const uint32_t b0 = word_of(f[ee][at / 4], at % 4), b1 = word_of(f[ee][at / 4], at % 4 + 1);
                        if (ks == 0) mma_k16(acc[ee], a[ee][ks], b0, b1);
                        else mma_k16_acc(acc[ee], a[ee][ks], b0, b1);
                    }
#pragma unroll
                for (int i = 0; i < 2; ++i)
#pragma unroll
                    for (int h = 0; h < 2; ++h) set_word(raw[4 * c + i + 2 * k][h], w, pack_bf16(acc[0][i + 2 * h], acc[1][i + 2 * h]));
            }
        }
        if (w == 1) mid();
    }
#pragma unroll
    for (int s = 0; s < 4 * KS; ++s) {
        const int u = 16 * (s / 4) + q + 4 * (s % 4);
        const uint32_t o = a0 + 32u * (uint32_t)u;
        if (u < U) {
            sts128(swz<K>(o), raw[s][0]);
            sts128(swz<K>(o + row8_off), raw[s][1]);
        }
    }
}

// The two phases that stay inside a box of 64 coordinates: contiguous blocks of eight, fa, and blocks over the eight chunks of a
// row, fb.  The rows of sixteen are this warp's, so that its own ordering is enough between the phases.
__device__ __forceinline__ void box_contiguous(const uint32_t (&fa)[8], uint32_t box, int lane) {
    const uint32_t row = box + 128u * (uint32_t)((lane & 7) + ((lane >> 3) & 1) * 8);
    const uint32_t hi = (uint32_t)lane >> 4, x = (row >> 7) & 7u;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        const uint32_t addr = row + (((2u * c + hi) ^ x) << 4);
        uint32_t a[4];
        ldmatrix_x4(a, addr);
        const uint32_t a_lo[2] = {a[0], a[1]}, a_hi[2] = {a[2], a[3]};
        float c0[4], c1[4];
        mma_k8(c0, a_lo, fa[2 * c]);
        mma_k8(c1, a_hi, fa[2 * c + 1]);
        stmatrix_x4(addr, pack_bf16(c0[0], c0[1]), pack_bf16(c0[2], c0[3]), pack_bf16(c1[0], c1[1]), pack_bf16(c1[2], c1[3]));
    }
}
__device__ __forceinline__ void box_octet(const uint32_t (&fb)[8], uint32_t box, int g, int q) {
    const uint32_t row = box + 128u * (uint32_t)g, x = (row >> 7) & 7u;
    uint4 raw[2][2];
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        const uint32_t addr = row + (((uint32_t)(2 * q + j) ^ x) << 4);
        raw[j][0] = lds128(addr);
        raw[j][1] = lds128(addr + 1024u);
    }
    octet_mma8(raw, fb);
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        const uint32_t addr = row + (((uint32_t)(2 * q + j) ^ x) << 4);
        sts128(addr, raw[j][0]);
        sts128(addr + 1024u, raw[j][1]);
    }
}

template <int K>
__global__ void __launch_bounds__(KindOf<K>::threads, 1)
harp_pipe_kernel(const __grid_constant__ CUtensorMap tmap, int32_t *err, const __grid_constant__ PipePass P) {
    constexpr bool LOWER = KindOf<K>::lower, B16 = KindOf<K>::b16;
    constexpr int LW = KindOf<K>::wide ? 32 : 16;          // upper: positions of a column group
    constexpr int KS = KindOf<K>::ks, TEAMS = KindOf<K>::teams, kTeamWarps = KindOf<K>::team_warps, kTeamThreads = KindOf<K>::team_threads;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ __align__(8) uint64_t full_bar[TEAMS * kMaxPipeBufs];
    __shared__ int dead;
    const uint32_t smem0 = (smem_u32(smem_raw) + 127u) & ~127u;
    const int team = threadIdx.x / kTeamThreads, tid = threadIdx.x - team * kTeamThreads;
    const int lane = tid & 31, warp = tid >> 5, g = lane >> 2, q = lane & 3;
    const int NB = P.n_buf;
    const uint32_t bufs = smem0 + (uint32_t)(team * NB * P.tile_bytes);
    const uint32_t bf_s = smem0 + (uint32_t)(TEAMS * NB * P.tile_bytes);
    const uint32_t tab_s = bf_s + 4u * (uint32_t)P.bfrag_words;
    for (int i = threadIdx.x; i < P.tables_len; i += TEAMS * kTeamThreads)
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(tab_s + 4u * i), "l"(P.tables + i) : "memory");
    if (threadIdx.x == 0) {
        for (int b = 0; b < TEAMS * kMaxPipeBufs; ++b) mbar_init(smem_u32(&full_bar[b]), 1);
        dead = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();

    // rows of a lane: LOWER g and g + 8 of a 16-row group; upper: g / 2 and g / 2 + 4 of the half g & 1
    const uint32_t row0_off = LOWER ? 128u * (uint32_t)g : (uint32_t)((g & 1) * P.box_pitch + (g >> 1) * P.row_bytes);
    const uint32_t row8_off = LOWER ? 1024u : 4u * (uint32_t)P.row_bytes;
    const uint32_t mt_step = LOWER ? 2048u : 8u * (uint32_t)P.row_bytes;

    // Rows past the end of the batch arrive as zeros and are not written.
    auto load = [&](int cg, int tile, int b) {
        const uint32_t bar = smem_u32(&full_bar[team * kMaxPipeBufs + b]), dst = bufs + (uint32_t)(b * P.tile_bytes);
        mbar_expect_tx(bar, (uint32_t)(P.n_box * P.box_bytes));
        for (int k = 0; k < P.n_box; ++k) {
            if constexpr (LOWER) harp_tm::tma_load_2d(dst + (uint32_t)(k * P.box_pitch), &tmap, 64 * (cg * P.n_box + k), tile * 16 * P.MT, bar);
            else tma_load_4d(dst + (uint32_t)(k * P.box_pitch), &tmap, LW * cg, 0, 0, tile * 16 * P.MT + 8 * P.MT * k, bar);
        }
    };
    auto store = [&](int cg, int tile, int b) {
        const uint32_t src = bufs + (uint32_t)(b * P.tile_bytes);
        for (int k = 0; k < P.n_box; ++k) {
            if constexpr (LOWER) harp_tm::tma_store_2d(&tmap, 64 * (cg * P.n_box + k), tile * 16 * P.MT, src + (uint32_t)(k * P.box_pitch));
            else tma_store_4d(&tmap, LW * cg, 0, 0, tile * 16 * P.MT + 8 * P.MT * k, src + (uint32_t)(k * P.box_pitch));
        }
        harp_tm::bulk_commit();
    };
    auto team_sync = [&]() { asm volatile("bar.sync %0, %1;" ::"r"(1 + team), "n"(kTeamThreads) : "memory"); };

    // segments of this CTA: a column group and its tiles
    int64_t at = 0, end = 1;
    if (P.n_parts == 0) {
        const int64_t all = (int64_t)P.n_cg * P.n_tiles, per = all / gridDim.x, extra = all % gridDim.x;
        at = blockIdx.x * per + min((int64_t)blockIdx.x, extra);
        end = at + per + ((int64_t)blockIdx.x < extra ? 1 : 0);
    }
    uint32_t parity = 0;
    bool waited = false;
    while (at < end) {
        int cg, first, step, count;
        if (P.n_parts > 0) {
            cg = blockIdx.x % P.n_cg;
            first = blockIdx.x / P.n_cg;
            step = P.n_parts;
            count = first < P.n_tiles ? (P.n_tiles - first + step - 1) / step : 0;
            at = end;
        } else {
            cg = (int)(at / P.n_tiles);
            first = (int)(at - (int64_t)cg * P.n_tiles);
            step = 1;
            count = (int)min((int64_t)(P.n_tiles - first), end - at);
            at += count;
        }
        // fragments of the column group (plan data); every team is through with the ones before
        __syncthreads();
        const uint32_t *src = P.bfrag + (size_t)cg * P.frag_stride;
        for (int i = threadIdx.x * 4; i < P.bfrag_words; i += TEAMS * kTeamThreads * 4) cp_async16(bf_s + 4u * i, src + P.smem_off + i);
        [[maybe_unused]] uint32_t fa[8], fb[8], wf[2][2][8];
        if constexpr (K == kUpper8Wide) {
            // the fragments of two neighbouring groups of sixteen positions: item = (block, octet of the 32 positions)
#pragma unroll
            for (int p = 0; p < 2; ++p)
#pragma unroll
                for (int k = 0; k < 2; ++k) {
                    const int i1 = min(warp + kTeamWarps * k, P.ph[p].n_items - 1), l8 = i1 & 3;
                    const uint4 *f = reinterpret_cast<const uint4 *>(src + (l8 >> 1) * (P.frag_stride / 2) + P.ph[p].bfrag_off + ((i1 >> 2) * 2 + (l8 & 1)) * 256) + lane;
                    const uint4 f0 = __ldg(f), f1 = __ldg(f + 32);
                    wf[p][k][0] = f0.x; wf[p][k][1] = f0.y; wf[p][k][2] = f0.z; wf[p][k][3] = f0.w;
                    wf[p][k][4] = f1.x; wf[p][k][5] = f1.y; wf[p][k][6] = f1.z; wf[p][k][7] = f1.w;
                }
        }
        if constexpr (LOWER) {
            const int box = min(warp, P.n_box - 1);
            const uint4 *f = reinterpret_cast<const uint4 *>(src + P.pair_off[1] + box * 256) + lane;
            const uint4 f0 = __ldg(f), f1 = __ldg(f + 32);
            fb[0] = f0.x; fb[1] = f0.y; fb[2] = f0.z; fb[3] = f0.w;
            fb[4] = f1.x; fb[5] = f1.y; fb[6] = f1.z; fb[7] = f1.w;
#pragma unroll
            for (int e = 0; e < 8; ++e) fa[e] = __ldg(src + P.pair_off[0] + (box * 8 + e) * 32 + lane);
        }
        if (!waited) {                               // the rows only once the kernel before has completed
            asm volatile("griddepcontrol.wait;" ::: "memory");
            asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
            waited = true;
        }
        if (tid == 0 && !*(volatile int *)&dead)
            for (int k = 0; k < NB; ++k)
                if (team + k * TEAMS < count) load(cg, first + (team + k * TEAMS) * step, k);
        cp_async_wait_all();
        __syncthreads();
        int b = 0;
        for (int t = team; t < count; t += TEAMS, b = b + 1 == NB ? 0 : b + 1) {
            const uint32_t bar = smem_u32(&full_bar[team * kMaxPipeBufs + b]), sbase = bufs + (uint32_t)(b * P.tile_bytes);
            uint32_t it = 0;
            while (!mbar_try(bar, (parity >> b) & 1u)) {
                if (++it > kPipeSpin || ((it & 63) == 63 && *(volatile int *)&dead)) {
                    *(volatile int *)&dead = 1;       // from here on nothing is copied any more
                    atomicExch(err, 301);
                    parity ^= 1u << b;        // (undone below: the phase is still awaited)
                    break;
                }
            }
            parity ^= 1u << b;
            // the store of the tile before has had a phase's time to be read: refill its buffer
            auto refill = [&]() {
                if (tid == 0 && t > team && t + (NB - 1) * TEAMS < count && !*(volatile int *)&dead) {
                    harp_tm::bulk_wait_read0();
                    load(cg, first + (t + (NB - 1) * TEAMS) * step, b == 0 ? NB - 1 : b - 1);
                }
            };
            if constexpr (K == kUpper8Wide) {
#pragma unroll
                for (int p = 0; p < 2; ++p) {
                    const PipePhase &ph = P.ph[p];
                    if (p > 0) team_sync();
                    uint32_t so[2];
                    bool ok[2];
#pragma unroll
                    for (int j = 0; j < 2; ++j) {
                        ok[j] = q + 4 * j < ph.B_real;
                        so[j] = ok[j] ? (uint32_t)((q + 4 * j) * ph.step[1]) : 0u;
                    }
#pragma unroll
                    for (int k = 0; k < 2; ++k) {
                        const int i1 = warp + kTeamWarps * k;
                        if (i1 < ph.n_items) {
                            const uint32_t a0 = sbase + lds32p(tab_s + 4u * (uint32_t)(ph.items_off + i1)) + row0_off;
                            uint4 raw[2][2];
                            uint32_t ad[2][2];
#pragma unroll
                            for (int j = 0; j < 2; ++j) {
                                ad[j][0] = swz<K>(a0 + so[j]);
                                ad[j][1] = swz<K>(a0 + so[j] + row8_off);
                                raw[j][0] = lds128(ad[j][0]);
                                raw[j][1] = lds128(ad[j][1]);
                            }
                            octet_mma8(raw, wf[p][k]);
#pragma unroll
                            for (int j = 0; j < 2; ++j)
                                if (ok[j]) {
                                    sts128(ad[j][0], raw[j][0]);
                                    sts128(ad[j][1], raw[j][1]);
                                }
                        }
                    }
                    if (p == 0) refill();
                }
            } else if constexpr (KS > 0) {
                dense_octet<K>(sbase + 16u * (uint32_t)warp + row0_off, row8_off, q, P.ph[0].B_real,
                                bf_s + 16u * (uint32_t)(warp * 8 * KS * KS * 32 + lane), refill);
            } else
            for (int p = 0; p < P.n_phases; ++p) {
                const PipePhase &ph = P.ph[p];
                if (p > 0) team_sync();
                if (LOWER && ph.mode == 0) {
                    if constexpr (LOWER) if (warp < P.n_box) {
                        uint32_t box = sbase + (uint32_t)(warp * P.box_pitch);
                        for (int mt = 0; mt < P.MT; ++mt, box += 2048u) {
                            if (P.pair_bwd) box_octet(fb, box, g, q);
                            else box_contiguous(fa, box, lane);
                            __syncwarp();
                            if (P.pair_bwd) box_contiguous(fa, box, lane);
                            else box_octet(fb, box, g, q);
                        }
                    }
                } else if constexpr (B16) {
                    uint32_t so[4];
                    bool ok[4];
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        ok[j] = ph.lm * q + ph.jr[j] < ph.B_real;
                        so[j] = ok[j] ? local_off(ph, ph.lm * q + ph.jr[j]) : 0u;      // padded slots read slot 0 and are not stored
                    }
                    const int n_work = ph.n_items * P.MT;
                    for (int w = warp; w < n_work; w += kTeamWarps) {
                        const int i1 = w >> P.mt_shift, mt = w & (P.MT - 1);
                        const uint32_t a0 = sbase + lds32p(tab_s + 4u * (uint32_t)(ph.items_off + i1)) + row0_off + (uint32_t)mt * mt_step;
                        const uint32_t bfa = bf_s + 4u * (uint32_t)(ph.bfrag_off + (i1 * 256 + lane) * 4);
                        uint4 raw[4][2], bf[8];
                        uint32_t unused[8][4];
#pragma unroll
                        for (int e = 0; e < 8; ++e) bf[e] = lds128(bfa + e * 512);
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            raw[j][0] = lds128(swz<K>(a0 + so[j]));
                            raw[j][1] = lds128(swz<K>(a0 + so[j] + row8_off));
                        }
                        octet_mma16<true>(raw, bf, unused);
#pragma unroll
                        for (int j = 0; j < 4; ++j)
                            if (ok[j]) {
                                sts128(swz<K>(a0 + so[j]), raw[j][0]);
                                sts128(swz<K>(a0 + so[j] + row8_off), raw[j][1]);
                            }
                    }
                } else {
                    uint32_t so[2];
                    bool ok[2];
#pragma unroll
                    for (int j = 0; j < 2; ++j) {
                        ok[j] = ph.lm * q + ph.jr[j] < ph.B_real;
                        so[j] = ok[j] ? local_off(ph, ph.lm * q + ph.jr[j]) : 0u;
                    }
                    const int n_work = ph.n_items * P.MT;
                    for (int w = warp; w < n_work; w += kTeamWarps) {
                        const int i1 = w >> P.mt_shift, mt = w & (P.MT - 1);
                        const uint32_t a0 = sbase + lds32p(tab_s + 4u * (uint32_t)(ph.items_off + i1)) + row0_off + (uint32_t)mt * mt_step;
                        const uint32_t bfa = bf_s + 4u * (uint32_t)(ph.bfrag_off + i1 * 256 + lane * 4);
                        uint4 raw[2][2];
                        uint32_t bf[8], ad[2][2];
#pragma unroll
                        for (int j = 0; j < 2; ++j) {
                            ad[j][0] = swz<K>(a0 + so[j]);
                            ad[j][1] = swz<K>(a0 + so[j] + row8_off);
                            raw[j][0] = lds128(ad[j][0]);
                            raw[j][1] = lds128(ad[j][1]);
                        }
                        {
                            const uint4 f0 = lds128(bfa), f1 = lds128(bfa + 512u);
                            bf[0] = f0.x; bf[1] = f0.y; bf[2] = f0.z; bf[3] = f0.w;
                            bf[4] = f1.x; bf[5] = f1.y; bf[6] = f1.z; bf[7] = f1.w;
                        }
                        octet_mma8(raw, bf);
#pragma unroll
                        for (int j = 0; j < 2; ++j)
                            if (ok[j]) {
                                sts128(ad[j][0], raw[j][0]);
                                sts128(ad[j][1], raw[j][1]);
                            }
                    }
                }
                if (p == 0) refill();
            }
            harp_tm::fence_async_smem();             // results before the copy engine reads them
            team_sync();
            if (tid == 0 && !*(volatile int *)&dead) {
                store(cg, first + t * step, b);
            }
        }
        if (tid == 0) harp_tm::bulk_wait_read0();
    }
    if (tid == 0) {
        harp_tm::bulk_wait0();
        if (*(volatile int *)&dead)
            ring_drain(parity, NB, kPipeSpin, [&](int k, uint32_t phase) { return mbar_try(smem_u32(&full_bar[team * kMaxPipeBufs + k]), phase); });
    }
}

// ------------------------------------------------------------------------------- host

typedef CUresult (*EncodeTiled)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *, const cuuint64_t *,
                                const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle,
                                CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

constexpr int kPipeSmem = 226 * 1024;

template <int K>
cudaError_t launch_pipe(const CUtensorMap &tmap, int32_t *err, const PipePass &P, unsigned grid, size_t smem, bool overlap, cudaStream_t stream) {
    const cudaError_t ae = cudaFuncSetAttribute(harp_pipe_kernel<K>, cudaFuncAttributeMaxDynamicSharedMemorySize, kPipeSmem);
    if (ae != cudaSuccess) return ae;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(KindOf<K>::threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = overlap ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, harp_pipe_kernel<K>, tmap, err, P);
}

// Fragments of the dense blocks (see dense_octet), sixteen positions per column group.
std::vector<uint32_t> dense_fragments(const harp_plan *plan, const GPhase &gp, int n_cg, int ks, int dir) {
    const int U = gp.B_real;
    std::vector<uint32_t> frag((size_t)n_cg * 16 * 4 * ks * ks * 32);
    std::vector<double> F;
    auto coord = [&](int slot) { return 16 * (slot / 16) + strided_slot(slot % 16, 16, 1); };
    for (int l = 0; l < 16 * n_cg; ++l) {
        fused_block(plan, HostPhase{gp.t0, gp.t1, U, gp.S, 0, 1}, l, F);
        auto G = [&](int slot_in, int slot_out) -> double {
            const int i = coord(slot_in), o = coord(slot_out);
            return i >= U || o >= U ? 0.0 : dir == 0 ? F[(size_t)i * U + o] : F[(size_t)o * U + i];
        };
        for (int c = 0; c < ks; ++c)
            for (int k = 0; k < 2; ++k)
                for (int s = 0; s < ks; ++s)
                    for (int h = 0; h < 2; ++h) {
                        const int f = 2 * (k * ks + s) + h;
                        // [octet][pair of positions][c][position of the pair][f / 4][lane][f % 4]
                        uint32_t *dst = frag.data() + ((size_t)(((l / 2) * ks + c) * 2 + l % 2) * ks + f / 4) * 128 + f % 4;
                        for (int lane = 0; lane < 32; ++lane) {
                            const int n = 16 * c + 8 * k + (lane >> 2), kk = 16 * s + 8 * h + 2 * (lane & 3);
                            dst[lane * 4] = f2bf(G(kk, n)) | ((uint32_t)f2bf(G(kk + 1, n)) << 16);
                        }
                    }
    }
    return frag;
}

}  // namespace

struct PipePlan {
    PipePass dir[2];           // forward, transpose
    int kind = kLower8;
    int64_t d = 0, S_mid = 1;
    int r_in = 1, r_out = 1;   // upper: radices of the inner and the outer digit of a tile
    int64_t s_in = 0, s_out = 0;   // ... and their strides in coordinates
    size_t smem = 0;
    int sms = 148;
    int32_t *d_err = nullptr;
    EncodeTiled encode = nullptr;
    std::vector<void *> dev_allocs;
};

void harp_pipe_destroy(PipePlan *pp) {
    if (!pp) return;
    for (void *p : pp->dev_allocs) cudaFree(p);
    delete pp;
}

// (1 to 32 rows of d = 5120 .. 28672: below nine rows the slab pass loses 0.2 us to the kernel of harp_split.cu, which reads only the
// rows it has, and so does the sixteen-wide upper pass up to one row tile; the others are ahead from the first row on.  The
// wide tiles of two phases pay once they give three quarters of the SMs one: 128 rows of d = 28672 14.0 -> 13.1 us, 256 of
// d = 14336 13.3 -> 12.3; at half of that 0.3 to 0.6 us are lost.)
int64_t harp_pipe_min_rows(const PipePlan *pp) {
    switch (pp->kind) {
        case kLower8: return 9;
        case kUpper16: return 17;
        case kUpper8Wide: return 16 * (3 * pp->sms / (4 * pp->dir[0].n_cg)) + 1;
        default: return 1;
    }
}

int32_t harp_pipe_error_word(const PipePlan *pp) {
    if (!pp || !pp->d_err) return 0;
    int32_t v = 0;
    return cudaMemcpy(&v, pp->d_err, sizeof(v), cudaMemcpyDeviceToHost) == cudaSuccess ? v : -1;
}

// The pass over `phs` (lower: slabs of S_mid coordinates; upper: sixteen neighbouring positions of all U slabs).
// HARP_ERR_UNSUPPORTED: a shape for which the layouts above are not free of conflicts, or whose tiles do not fit.
harp_status_t harp_pipe_build(const harp_plan *plan, const std::vector<GPhase> &phs, bool lower, int64_t S_mid, int64_t U, bool wide, const PassFrags &fr,
                              PipePlan **out) {
    *out = nullptr;
    const int np = (int)phs.size(), pair = lower ? 2 : 0;     // lower: the first two phases count as one
    if (np < 1 || np > kMaxPipePhases || !harp_tensor_map_encoder(plan)) return HARP_ERR_UNSUPPORTED;
    int widest = 8;
    for (const GPhase &gp : phs) widest = std::max(widest, gp.B);
    PipePass P{};
    PipePlan pl;
    pl.kind = lower ? kLower8 : widest == 8 ? (wide ? kUpper8Wide : np == 1 && S_mid % 32 == 0 ? kUpper8One : kUpper8) : widest == 16 ? kUpper16 : widest == 32 ? kDense32 : kDense48;
    const int ks = pl.kind >= kDense32 ? widest / 16 : 0, Lw = is_wide(pl.kind) ? 32 : 16;
    // Tiles of 32 positions read the fragments of two groups of sixteen as they lie in the plan, phases within groups: what the
    // kernel's item numbers mean for one phase only (kUpper8Wide finds them by group)
    if (wide ? pl.kind != kUpper8Wide || np != 2 : is_wide(pl.kind) && np != 1) return HARP_ERR_UNSUPPORTED;
    P.n_phases = lower ? np - 1 : np;
    if (lower) {
        if (np < 2 || S_mid > 512 || phs[0].B_real != 8 || phs[1].B_real != 8) return HARP_ERR_UNSUPPORTED;
        for (int p = 2; p < np; ++p)
            if (phs[(size_t)p].B != 8) return HARP_ERR_UNSUPPORTED;
        P.n_cg = (int)U;
        P.n_box = (int)(S_mid / 64);
    } else {
        // the digit of odd radix inside, so that a step of either digit is an odd number of columns
        if (np > (ks ? 1 : 2) || widest > 48 || S_mid % Lw != 0 || U > 64) return HARP_ERR_UNSUPPORTED;
        const int in = np == 2 && phs[1].B_real % 2 != 0 ? 1 : 0;
        if (np == 2 && phs[(size_t)in].B_real % 2 == 0) return HARP_ERR_UNSUPPORTED;
        pl.r_in = phs[(size_t)in].B_real;
        pl.s_in = phs[(size_t)in].S;
        if (np == 2) { pl.r_out = phs[(size_t)(1 - in)].B_real; pl.s_out = phs[(size_t)(1 - in)].S; }
        P.n_cg = (int)(S_mid / Lw);
        P.n_box = 2;
        P.row_bytes = (int32_t)(2 * Lw * U);
    }
    auto place = [&](int64_t c) -> int64_t {             // byte offset of an octet; c: coordinate within the slab (lower) or natural coordinate
        if (lower) return (c / 64) * P.box_pitch + (c % 64) * 2;
        const int64_t i = (c / pl.s_in) % pl.r_in, o = np == 2 ? (c / pl.s_out) % pl.r_out : 0;
        return (o * pl.r_in + i) * 2 * Lw + (c % Lw) * 2;
    };
    int words = ks ? 16 * 4 * ks * ks * 32 : 0, items = 0;
    for (int p = pair; p < np && !ks; ++p) {
        const int n_blk = (int)((lower ? S_mid : U * Lw) / phs[(size_t)p].B_real);
        if (fr.lm[p] != (lower ? 2 : 1)) return HARP_ERR_UNSUPPORTED;
        words += n_blk * (phs[(size_t)p].B == 16 ? 128 : 32);
        items += n_blk / 8;
    }
    if (!ks && !lower && words != fr.words * (Lw / 16)) return HARP_ERR_UNSUPPORTED;
    // the largest tile that fits; a pass of one phase refills a buffer while two others are full
    const int teams = wide ? 1 : pl.kind == kUpper16 ? 2 : 3;
    P.n_buf = wide || (np == 1 && !ks && !lower) ? 3 : 2;
    if (wide) words = 0;
    for (P.MT = ks || wide ? 1 : 4, P.mt_shift = P.MT / 2;; P.MT /= 2, --P.mt_shift) {
        P.box_bytes = lower ? 128 * 16 * P.MT : 8 * P.MT * P.row_bytes;
        P.box_pitch = P.box_bytes + (Lw == 32 ? 256 : 128);  // (P.box_bytes is a multiple of twice that)
        P.tile_bytes = P.n_box * P.box_pitch;
        pl.smem = (size_t)teams * P.n_buf * P.tile_bytes + (size_t)words * 4 + (size_t)items * 4 + 128;
        if (pl.smem <= kPipeSmem) break;
        if (P.MT == 1) return HARP_ERR_UNSUPPORTED;
    }
    pl.d = plan->d;
    pl.encode = reinterpret_cast<EncodeTiled>(harp_tensor_map_encoder(plan));
    pl.S_mid = S_mid;
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (sms > 0) pl.sms = sms;

    static const int jo16[4] = {0, 4, 8, 12}, jo8[2][2] = {{0, 4}, {0, 1}};
    harp_status_t st = HARP_OK;
    auto upload = [&](const auto &v) -> void * {
        const size_t bytes = v.size() * sizeof(v[0]);
        void *p = nullptr;
        if (st != HARP_OK) return nullptr;
        if (cudaMalloc(&p, std::max<size_t>(16, bytes)) != cudaSuccess) { st = HARP_ERR_ALLOC; return nullptr; }
        pl.dev_allocs.push_back(p);
        if (cudaMemcpy(p, v.data(), bytes, cudaMemcpyHostToDevice) != cudaSuccess) st = HARP_ERR_CUDA;
        return p;
    };
    pl.d_err = static_cast<int32_t *>(upload(std::vector<int32_t>(1, 0)));
    for (int dir = 0; dir < 2 && st == HARP_OK; ++dir) {
        std::vector<int32_t> tab;
        const int n_strided = np - pair;
        P.smem_off = lower && np > 2 ? fr.off[dir][dir == 0 ? 2 : np - 1] : 0;
        P.pair_bwd = dir;
        for (int p = 0; p < pair; ++p) P.pair_off[p] = fr.off[dir][p];
        for (int k = 0; k < P.n_phases; ++k) P.ph[k] = PipePhase{};          // mode 0
        for (int k = 0; k < n_strided; ++k) {
            const int p = dir == 0 ? pair + k : np - 1 - k;
            const GPhase &gp = phs[(size_t)p];
            PipePhase &D = P.ph[lower && dir == 0 ? k + 1 : k];
            D.mode = 1;
            D.B = gp.B;
            D.B_real = gp.B_real;
            if (ks) break;
            D.lm = lower ? 2 : 1;
            for (int j = 0; j < 4; ++j) D.jr[j] = gp.B == 16 ? jo16[j] : j < 2 ? jo8[D.lm - 1][j] : 0;
            D.items_off = (int32_t)tab.size();
            D.bfrag_off = fr.off[dir][p] - P.smem_off;
            if (lower) {                                 // in octets: eight to a box
                D.unit = (int32_t)(gp.S / 8);
                D.shift = 3;
                D.step[0] = 16;
                D.step[1] = P.box_pitch;
            } else {
                D.unit = 1;
                D.step[1] = (gp.S == pl.s_in ? 2 : 2 * pl.r_in) * Lw;
            }
            // octets of blocks, in the order of their fragments (upper: within position group 0)
            const int64_t span = gp.S * gp.B_real, all = lower ? S_mid : plan->d, lo_step = lower ? 8 : S_mid;
            for (int64_t hi = 0; hi < all; hi += span)
                for (int64_t lo = 0; lo < gp.S; lo += lo_step)
                    for (int64_t l8 = 0; l8 < (lower ? 8 : Lw); l8 += 8) {
                        const int64_t c = hi + lo + l8;
                        for (int r = 0; r < gp.B_real; ++r) {       // every octet that the kernel reaches
                            const int e = r * D.unit;
                            const int64_t a = place(c) + (e >> D.shift) * D.step[1] + (e & ((1 << D.shift) - 1)) * D.step[0];
                            if (a != place(c + r * gp.S) || a < 0 || a + 16 > (lower ? P.tile_bytes : P.row_bytes)) return HARP_ERR_UNSUPPORTED;
                        }
                        tab.push_back((int32_t)place(c));
                    }
            D.n_items = (int32_t)tab.size() - D.items_off;
            if (wide ? D.n_items > 32 : D.bfrag_off < 0 || D.bfrag_off + D.n_items * (gp.B == 16 ? 1024 : 256) > words) return HARP_ERR_UNSUPPORTED;
        }
        if ((int)tab.size() != items || words % 4 != 0) return HARP_ERR_UNSUPPORTED;
        P.tables_len = items;
        P.bfrag_words = words;
        P.tables = static_cast<const int32_t *>(upload(tab));
        P.frag_stride = wide ? 2 * fr.words : lower ? fr.words : words;
        P.bfrag = ks ? static_cast<const uint32_t *>(upload(dense_fragments(plan, phs[0], P.n_cg, ks, dir))) : fr.bfrag[dir];
        pl.dir[dir] = P;
    }
    PipePlan *pp = st == HARP_OK ? new (std::nothrow) PipePlan(pl) : nullptr;
    if (!pp) {
        for (void *p : pl.dev_allocs) cudaFree(p);
        return st == HARP_OK ? HARP_ERR_ALLOC : st;
    }
    *out = pp;
    return HARP_OK;
}

// x: n_rows contiguous rows, 16-byte aligned.
harp_status_t harp_pipe_apply(const PipePlan *pp, void *x, int64_t n_rows, int transpose, bool overlap, cudaStream_t stream) {
    if (!pp || n_rows > ((int64_t)1 << 30)) return HARP_ERR_UNSUPPORTED;
    PipePass P = pp->dir[transpose ? 1 : 0];
    const int64_t slots = pp->sms;
    // a batch with less than half a tile per CTA is cut finer
    while (P.MT > 1 && (n_rows + 16 * P.MT - 1) / (16 * P.MT) * P.n_cg * 2 < slots) {
        P.MT /= 2;
        --P.mt_shift;
        P.box_bytes /= 2;
    }
    P.n_tiles = (int32_t)((n_rows + 16 * P.MT - 1) / (16 * P.MT));
    // A column group per CTA keeps its fragments, and the CTAs at the same rows: neighbouring 32-byte runs meet in L2.  Where
    // the groups leave more than a tenth of the SMs without work, lower passes (whole lines) share the list out evenly.
    P.n_parts = (int32_t)std::min<int64_t>(P.n_tiles, std::max<int64_t>(1, slots / P.n_cg));
    if (pp->kind == kLower8 && (P.n_cg > slots || slots % P.n_cg * 10 > slots)) P.n_parts = 0;
    const unsigned grid = (unsigned)(P.n_parts > 0 ? (int64_t)P.n_parts * P.n_cg : std::min<int64_t>((int64_t)P.n_tiles * P.n_cg, slots));
    const EncodeTiled enc = pp->encode;
    CUtensorMap tmap = {};
    const cuuint32_t ones[4] = {1, 1, 1, 1};
    const cuuint64_t n = (cuuint64_t)n_rows, pitch = (cuuint64_t)pp->d * 2;
    CUresult r;
    if (pp->kind == kLower8) {
        const cuuint64_t gdim[2] = {(cuuint64_t)pp->d, n}, gstr[1] = {pitch};
        const cuuint32_t box[2] = {64, (cuuint32_t)(16 * P.MT)};
        r = enc(&tmap, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, x, gdim, gstr, box, ones, CU_TENSOR_MAP_INTERLEAVE_NONE,
                CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    } else {
        // (position, inner digit, outer digit, row)
        const cuuint64_t gdim[4] = {(cuuint64_t)pp->S_mid, (cuuint64_t)pp->r_in, (cuuint64_t)pp->r_out, n};
        const cuuint64_t gstr[3] = {(cuuint64_t)pp->s_in * 2, (cuuint64_t)(pp->r_out > 1 ? pp->s_out : pp->s_in) * 2, pitch};
        const cuuint32_t box[4] = {(cuuint32_t)(is_wide(pp->kind) ? 32 : 16), (cuuint32_t)pp->r_in, (cuuint32_t)pp->r_out, (cuuint32_t)(8 * P.MT)};
        r = enc(&tmap, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, x, gdim, gstr, box, ones, CU_TENSOR_MAP_INTERLEAVE_NONE,
                is_wide(pp->kind) ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_32B, CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    }
    if (r != CUDA_SUCCESS) return HARP_ERR_CUDA;
    cudaError_t err = cudaErrorInvalidValue;
    switch (pp->kind) {
        case kLower8: err = launch_pipe<kLower8>(tmap, pp->d_err, P, grid, pp->smem, overlap, stream); break;
        case kUpper8: err = launch_pipe<kUpper8>(tmap, pp->d_err, P, grid, pp->smem, overlap, stream); break;
        case kUpper8One: err = launch_pipe<kUpper8One>(tmap, pp->d_err, P, grid, pp->smem, overlap, stream); break;
        case kUpper8Wide: err = launch_pipe<kUpper8Wide>(tmap, pp->d_err, P, grid, pp->smem, overlap, stream); break;
        case kUpper16: err = launch_pipe<kUpper16>(tmap, pp->d_err, P, grid, pp->smem, overlap, stream); break;
        case kDense32: err = launch_pipe<kDense32>(tmap, pp->d_err, P, grid, pp->smem, overlap, stream); break;
        case kDense48: err = launch_pipe<kDense48>(tmap, pp->d_err, P, grid, pp->smem, overlap, stream); break;
    }
    g_harp_launches.fetch_add(1, std::memory_order_relaxed);
    return err == cudaSuccess && cudaGetLastError() == cudaSuccess ? HARP_OK : HARP_ERR_CUDA;
}
