// fp32 rows of any width: passes over column groups on CUDA cores.  This file chooses the passes and launches them; their kernels are
// harp_regs.cu's (radices up to 8 and pairs of 16, block kernels in registers), harp_big.cu's (one stage of radix 17 to 48) and, for all
// other shapes, the one below.
//
// A pass runs the consecutive stages [t0, t1) of the plan.  They mix coordinates at strides
// S, ..., S*E/b (S = stride of stage t0, E = product of the radices), so a column group of E * L
// coordinates -- L neighbouring positions below the stride S, in each of the E places -- is closed
// under the pass and its block kernels are small enough to stay in shared memory.  A CTA takes a
// column group, loads its block kernels once and walks over tiles of R = 32 * RT rows; the rows of a
// batch cross HBM once per pass (two passes up to d of about 30 k).
//
// A lane owns RT rows of the tile and a warp a block, so a block's kernel is the same for all 32 lanes
// (broadcast 16-byte loads).  Two tile layouts, both free of bank conflicts:
//   ROWS, RUNS  [row][coordinate], rows an odd number of 16-byte units apart: a lane reads four neighbouring coordinates of
//         its row at once (four neighbouring blocks of a strided stage).  ROWS: stages from stride 1 on, the tile is one
//         run of E coordinates per row; RUNS: stages at larger strides, E runs of L coordinates.
//   COLS  [coordinate][column], down the columns of a row-major matrix: the batch is the contiguous direction, so the
//         two-sided product of an fp32 matrix needs neither a transposed copy nor scratch.
// ROWS and COLS tiles move by bulk copies over three buffers: one SM moves about 30 bytes per cycle to and from L2, and
// a warp that issues loads and stores is held at that rate with every shared-memory access behind it (the arithmetic of a
// tile took four times as long with the copies done by extra warps through the load/store unit).  RUNS tiles (runs of
// 16 to 128 bytes) move by cp.async, the next tile under the arithmetic of this one.
#include <algorithm>
#include <new>

#include "harp_internal.h"
#include "harp_permute.h"
#include "harp_regs.h"
#include "harp_ring.h"
#include "harp_tm_ptx.cuh"

namespace {

using harp_tm::smem_u32;

constexpr int kWarps = 16;
constexpr int kF32Threads = 32 * kWarps;
constexpr int kMaxF32Phases = 12;
constexpr int kMaxF32Passes = 12;
constexpr int kMaxF32Radix = 64;
constexpr int kMaxBuf = 3;
constexpr uint32_t kF32Spin = 1u << 22;       // limit of every wait for a bulk copy

enum { ROWS = 0, RUNS = 1, COLS = 2 };

struct F32Phase {
    int32_t b, ls;             // radix, stride in units of the pass's own index e
    int32_t n_blk;             // blocks of the tile
    int32_t pitch;             // floats per row of a block kernel in shared memory
    int32_t w_off;             // float offset of the phase's block kernels
    int32_t base_off;          // tables: tile coordinate of every block's first entry
    int32_t pair;              // 1: runs together with the next phase (two radix-4 stages), 2: is that next phase
    int64_t k_off;             // offset of the stage in the plan's block array
};

struct F32Pass {
    int32_t n_ph, E, L, RT, mode;
    int32_t n_lo;              // groups of L positions below the stride (S / L)
    int32_t n_cg;              // column groups
    int32_t pitch;             // floats per tile row (ROWS) or tile coordinate
    int32_t tile_floats, n_buf;
    int32_t w_floats;          // block kernels of a column group
    int32_t smem;              // bytes
    int32_t big;               // has a radix above 16
    int32_t n_box, box_e;      // bulk copies of a tile; places (COLS) or runs of 32 coordinates (ROWS) one of them covers
    int64_t S, d;
    F32Phase ph[kMaxF32Phases];
    RegPass reg;               // shape > 0: the pass is one of harp_regs.cu or harp_big.cu and nothing above counts
};

__device__ __forceinline__ void cp_async4(float *dst, const float *src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async16(float *dst, const float *src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}

// two packed fp32 values and the packed fused multiply-add (each half rounds like fmaf)
struct F2 {
    unsigned long long v;
    __device__ __forceinline__ F2() {}
    __device__ __forceinline__ F2(float lo, float hi) { asm("mov.b64 %0, {%1, %2};" : "=l"(v) : "f"(lo), "f"(hi)); }
    __device__ __forceinline__ void fma(const F2 &a, const F2 &b) { asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(v) : "l"(a.v), "l"(b.v)); }
    __device__ __forceinline__ float lo() const { return __uint_as_float((uint32_t)v); }
    __device__ __forceinline__ float hi() const { return __uint_as_float((uint32_t)(v >> 32)); }
};

// one row of a block kernel (B entries, PITCH floats apart from the next)
template <int B> struct KRow {
    static constexpr int pitch = B == 2 ? 2 : (B + 3) / 4 * 4;
    float v[pitch];
    __device__ __forceinline__ void load(const float *p) {
        if constexpr (B == 2) {
            const float2 q = *reinterpret_cast<const float2 *>(p);
            v[0] = q.x; v[1] = q.y;
        } else {
#pragma unroll
            for (int j = 0; j < pitch; j += 4) {
                const float4 q = *reinterpret_cast<const float4 *>(p + j);
                v[j] = q.x; v[j + 1] = q.y; v[j + 2] = q.z; v[j + 3] = q.w;
            }
        }
    }
};

// out[j][u] = sum_i in[i][u] K[i][j], in place; u runs over the lane's rows
template <int B, int RT>
__device__ __forceinline__ void block_product(float (&in)[B][RT], const float *kw) {
    float acc[B][RT];
#pragma unroll
    for (int i = 0; i < B; ++i) {
        KRow<B> row;
        row.load(kw + i * KRow<B>::pitch);
#pragma unroll
        for (int j = 0; j < B; ++j)
#pragma unroll
            for (int u = 0; u < RT; ++u) acc[j][u] = i == 0 ? in[0][u] * row.v[j] : fmaf(in[i][u], row.v[j], acc[j][u]);
    }
#pragma unroll
    for (int j = 0; j < B; ++j)
#pragma unroll
        for (int u = 0; u < RT; ++u) in[j][u] = acc[j][u];
}

template <int RT> struct RowVec;
template <> struct RowVec<1> {
    static __device__ __forceinline__ void ld(const float *p, float (&v)[1]) { v[0] = *p; }
    static __device__ __forceinline__ void st(float *p, const float (&v)[1]) { *p = v[0]; }
};
template <> struct RowVec<2> {
    static __device__ __forceinline__ void ld(const float *p, float (&v)[2]) {
        const float2 q = *reinterpret_cast<const float2 *>(p);
        v[0] = q.x; v[1] = q.y;
    }
    static __device__ __forceinline__ void st(float *p, const float (&v)[2]) { *reinterpret_cast<float2 *>(p) = make_float2(v[0], v[1]); }
};

// ------------------------------------------------------------------ phases on [coordinate][column] tiles

template <int B, int RT>
__device__ __forceinline__ void col_phase(float *tile, const float *w, const int32_t *bases, const F32Phase &ph, int L, int warp, int lane) {
    const int step = ph.ls * L * 32 * RT;
    for (int k = warp; k < ph.n_blk; k += kWarps) {
        float *p = tile + bases[k] * 32 * RT + RT * lane;
        float in[B][RT];
#pragma unroll
        for (int i = 0; i < B; ++i) RowVec<RT>::ld(p + i * step, in[i]);
        block_product<B, RT>(in, w + k * (B * KRow<B>::pitch));
#pragma unroll
        for (int j = 0; j < B; ++j) RowVec<RT>::st(p + j * step, in[j]);
    }
}

// radix above 16 (at most 8 * NC): two warps share a block, each with half of its results in registers (neighbouring results of
// a row or column in a packed pair); operands and kernel rows are streamed, the next ones fetched while these are
// multiplied.  Nobody stores before everybody has read.  COLS tiles hold a lane's columns next to each other; in RUNS
// tiles a lane reads its row one coordinate at a time (four wavefronts, as many as for 16 bytes a lane).
template <int NC, int RT, int MODE>
__device__ __forceinline__ void phase_large(float *tile, int pitch, const float *w, const int32_t *bases, const F32Phase &ph, int L, int warp, int lane) {
    constexpr int H = 4 * NC;
    const int step = ph.ls * L * (MODE == COLS ? 32 * RT : 1), b = ph.b, j0 = (warp & 1) * H;
    for (int k0 = 0; k0 < ph.n_blk; k0 += kWarps / 2) {
        const int k = k0 + (warp >> 1);
        const bool have = k < ph.n_blk;
        const int base = have ? bases[k] : 0;
        float *p = MODE == COLS ? tile + base * 32 * RT + RT * lane : tile + lane * pitch + base;
        auto get = [&](const float *q, float (&v)[RT]) {
            if constexpr (MODE == COLS) {
                RowVec<RT>::ld(q, v);
            } else {
                v[0] = q[0];
                if constexpr (RT == 2) v[RT - 1] = q[32 * pitch];
            }
        };
        F2 acc[H / 2][RT];
#pragma unroll
        for (int j = 0; j < H / 2; ++j)
#pragma unroll
            for (int u = 0; u < RT; ++u) acc[j][u].v = 0;
        if (have) {
            const float *kw = w + k * (b * 8 * NC) + j0;
            const float *pi = p;
            float v[RT];
            get(pi, v);
#pragma unroll 2
            for (int i = 0; i < b; ++i, kw += 8 * NC) {
                F2 vv[RT];
#pragma unroll
                for (int u = 0; u < RT; ++u) vv[u] = F2(v[u], v[u]);
                pi += i + 1 < b ? step : 0;
                get(pi, v);
#pragma unroll
                for (int j = 0; j < H; j += 4) {
                    const float4 q = *reinterpret_cast<const float4 *>(kw + j);
                    const F2 q0(q.x, q.y), q1(q.z, q.w);
#pragma unroll
                    for (int u = 0; u < RT; ++u) {
                        acc[j / 2][u].fma(vv[u], q0);
                        acc[j / 2 + 1][u].fma(vv[u], q1);
                    }
                }
            }
        }
        __syncthreads();
        if (have) {
#pragma unroll
            for (int j = 0; j < H; ++j)
                if (j0 + j < b) {
                    float o[RT];
#pragma unroll
                    for (int u = 0; u < RT; ++u) o[u] = (j & 1) ? acc[j / 2][u].hi() : acc[j / 2][u].lo();
                    float *q = p + (j0 + j) * step;
                    if constexpr (MODE == COLS) {
                        RowVec<RT>::st(q, o);
                    } else {
                        q[0] = o[0];
                        if constexpr (RT == 2) q[32 * pitch] = o[RT - 1];
                    }
                }
        }
    }
}

// Two consecutive radix-4 stages on sixteen coordinates held in registers ([second digit][first digit]): half the operand
// traffic of two phases.  w1, w2: kernel of the unit's first block in either stage; the unit's blocks are s1 apart.
template <int RT>
__device__ __forceinline__ void product_4x4(float (&v)[4][4][RT], const float *w1, const float *w2, int s1, int transpose) {
    auto first = [&]() {
#pragma unroll
        for (int i2 = 0; i2 < 4; ++i2) block_product<4, RT>(v[i2], w1 + i2 * s1 * 16);
    };
    auto second = [&]() {
#pragma unroll
        for (int i1 = 0; i1 < 4; ++i1) {
            float c[4][RT];
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int u = 0; u < RT; ++u) c[i][u] = v[i][i1][u];
            block_product<4, RT>(c, w2 + i1 * s1 * 16);
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int u = 0; u < RT; ++u) v[i][i1][u] = c[i][u];
        }
    };
    if (!transpose) { first(); second(); } else { second(); first(); }
}

// unit (a, r, l) of a pair of phases: its blocks in either stage are numbers ((4 a + i) ls + r) L + l
template <int RT>
__device__ __forceinline__ void col_phase_4x4(float *tile, const float *w1, const float *w2, const F32Phase &ph, int L, int transpose, int warp, int lane) {
    const int s1 = ph.ls * L, p1 = s1 * 32 * RT;
    for (int u0 = warp; u0 < ph.n_blk / 4; u0 += kWarps) {
        const int a = u0 / s1, rl = u0 - a * s1;
        float *p = tile + (a * 16 * s1 + rl) * 32 * RT + RT * lane;
        const int k0 = 4 * a * s1 + rl;
        float v[4][4][RT];
#pragma unroll
        for (int i = 0; i < 16; ++i) RowVec<RT>::ld(p + i * p1, v[i >> 2][i & 3]);
        product_4x4<RT>(v, w1 + k0 * 16, w2 + k0 * 16, s1, transpose);
#pragma unroll
        for (int i = 0; i < 16; ++i) RowVec<RT>::st(p + i * p1, v[i >> 2][i & 3]);
    }
}

// ------------------------------------------------------------------ phases on [row][coordinate] tiles (a lane's rows: lane, lane + 32)

__device__ __forceinline__ float comp(const float4 &q, int c) { return c == 0 ? q.x : c == 1 ? q.y : c == 2 ? q.z : q.w; }
__device__ __forceinline__ void set_comp(float4 &q, int c, float v) { if (c == 0) q.x = v; else if (c == 1) q.y = v; else if (c == 2) q.z = v; else q.w = v; }

// 16-byte chunk ch (coordinates 4 ch .. 4 ch + 3) of a lane's row `lane + 32 u`.  ROWS: boxes of 32 coordinates x R rows as the
// copy engine writes them, 128-byte rows with the chunk index XORed by the row (mod 8); RUNS: rows of `pitch` floats.
template <int RT, int MODE>
__device__ __forceinline__ float *rm_chunk(float *tile, int pitch, int lane, int u, int ch) {
    if constexpr (MODE == ROWS) return tile + (ch >> 3) * (32 * RT * 32) + (lane + 32 * u) * 32 + (((ch ^ lane) & 7) << 2);
    else return tile + (lane + 32 * u) * pitch + 4 * ch;
}

// contiguous blocks of 4, 8 or 16 coordinates
template <int B, int RT>
__device__ __forceinline__ void rm_contig(float *tile, const float *w, int n_blk, int warp, int lane) {
    for (int k = warp; k < n_blk; k += kWarps) {
        float in[B][RT];
#pragma unroll
        for (int u = 0; u < RT; ++u)
#pragma unroll
            for (int j = 0; j < B; j += 4) {
                const float4 q = *reinterpret_cast<const float4 *>(rm_chunk<RT, ROWS>(tile, 0, lane, u, (k * B + j) >> 2));
                in[j][u] = q.x; in[j + 1][u] = q.y; in[j + 2][u] = q.z; in[j + 3][u] = q.w;
            }
        block_product<B, RT>(in, w + k * (B * KRow<B>::pitch));
#pragma unroll
        for (int u = 0; u < RT; ++u)
#pragma unroll
            for (int j = 0; j < B; j += 4)
                *reinterpret_cast<float4 *>(rm_chunk<RT, ROWS>(tile, 0, lane, u, (k * B + j) >> 2)) = make_float4(in[j][u], in[j + 1][u], in[j + 2][u], in[j + 3][u]);
    }
}

template <int RT>
__device__ __forceinline__ void rm_contig_4x4(float *tile, const float *w1, const float *w2, int n_units, int transpose, int warp, int lane) {
    for (int k = warp; k < n_units; k += kWarps) {
        float v[4][4][RT];
#pragma unroll
        for (int u = 0; u < RT; ++u)
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const float4 q = *reinterpret_cast<const float4 *>(rm_chunk<RT, ROWS>(tile, 0, lane, u, 4 * k + j));
                v[j][0][u] = q.x; v[j][1][u] = q.y; v[j][2][u] = q.z; v[j][3][u] = q.w;
            }
        product_4x4<RT>(v, w1 + k * 64, w2 + k * 64, 1, transpose);
#pragma unroll
        for (int u = 0; u < RT; ++u)
#pragma unroll
            for (int j = 0; j < 4; ++j)
                *reinterpret_cast<float4 *>(rm_chunk<RT, ROWS>(tile, 0, lane, u, 4 * k + j)) = make_float4(v[j][0][u], v[j][1][u], v[j][2][u], v[j][3][u]);
    }
}

// strided blocks (stride a multiple of 4): four neighbouring blocks at once
template <int B, int RT, int MODE>
__device__ __forceinline__ void rm_quad(float *tile, int pitch, const float *w, const int32_t *bases, const F32Phase &ph, int L, int warp, int lane) {
    const int step = (ph.ls * L) >> 2;
    // above radix 8 the operands of two rows do not fit the registers: one row at a time
    constexpr int U = B > 8 ? 1 : RT;
    for (int k = 4 * warp; k < ph.n_blk; k += 4 * kWarps)
#pragma unroll 1
        for (int h = 0; h < RT / U; ++h) {
            const int ch = bases[k] >> 2;
            float4 in[B][U];
#pragma unroll
            for (int i = 0; i < B; ++i)
#pragma unroll
                for (int u = 0; u < U; ++u) in[i][u] = *reinterpret_cast<const float4 *>(rm_chunk<RT, MODE>(tile, pitch, lane, h + u, ch + i * step));
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                float one[B][U];
#pragma unroll
                for (int i = 0; i < B; ++i)
#pragma unroll
                    for (int u = 0; u < U; ++u) one[i][u] = comp(in[i][u], c);
                block_product<B, U>(one, w + (k + c) * (B * KRow<B>::pitch));
#pragma unroll
                for (int i = 0; i < B; ++i)
#pragma unroll
                    for (int u = 0; u < U; ++u) set_comp(in[i][u], c, one[i][u]);
            }
#pragma unroll
            for (int i = 0; i < B; ++i)
#pragma unroll
                for (int u = 0; u < U; ++u) *reinterpret_cast<float4 *>(rm_chunk<RT, MODE>(tile, pitch, lane, h + u, ch + i * step)) = in[i][u];
        }
}

// any stride, one coordinate at a time
template <int B, int RT>
__device__ __forceinline__ void rm_scalar(float *tile, const float *w, const int32_t *bases, const F32Phase &ph, int L, int warp, int lane) {
    const int step = ph.ls * L;
    for (int k = warp; k < ph.n_blk; k += kWarps) {
        const int c0 = bases[k];
        auto at = [&](int i, int u) { const int c = c0 + i * step; return rm_chunk<RT, ROWS>(tile, 0, lane, u, c >> 2) + (c & 3); };
        float in[B][RT];
#pragma unroll
        for (int i = 0; i < B; ++i)
#pragma unroll
            for (int u = 0; u < RT; ++u) in[i][u] = *at(i, u);
        block_product<B, RT>(in, w + k * (B * KRow<B>::pitch));
#pragma unroll
        for (int i = 0; i < B; ++i)
#pragma unroll
            for (int u = 0; u < RT; ++u) *at(i, u) = in[i][u];
    }
}

template <int B, int RT, int MODE>
__device__ __forceinline__ void phase_b(float *tile, int pitch, const float *w, const int32_t *bases, const F32Phase &ph, int L, int warp, int lane) {
    if constexpr (MODE == COLS) {
        col_phase<B, RT>(tile, w, bases, ph, L, warp, lane);
    } else {
        if ((ph.ls * L) % 4 == 0) { rm_quad<B, RT, MODE>(tile, pitch, w, bases, ph, L, warp, lane); return; }
        if constexpr (MODE == ROWS) {
            if constexpr (B == 4 || B == 8 || B == 16)
                if (ph.ls == 1) { rm_contig<B, RT>(tile, w, ph.n_blk, warp, lane); return; }
            rm_scalar<B, RT>(tile, w, bases, ph, L, warp, lane);
        }
    }
}

template <int RT, int MODE, bool BIG>
__device__ __forceinline__ void run_phase(float *tile, int pitch, const float *w, const int32_t *bases, const F32Phase &ph, int L, int warp, int lane) {
#define HARP_F32_CASE(B) case B: phase_b<B, RT, MODE>(tile, pitch, w, bases, ph, L, warp, lane); return
    switch (ph.b) {
        HARP_F32_CASE(2); HARP_F32_CASE(3); HARP_F32_CASE(4); HARP_F32_CASE(5); HARP_F32_CASE(6); HARP_F32_CASE(7); HARP_F32_CASE(8);
        default: break;
    }
    if constexpr (!BIG) {
        switch (ph.b) {
            HARP_F32_CASE(9); HARP_F32_CASE(10); HARP_F32_CASE(11); HARP_F32_CASE(12); HARP_F32_CASE(13); HARP_F32_CASE(14); HARP_F32_CASE(15);
            default: phase_b<16, RT, MODE>(tile, pitch, w, bases, ph, L, warp, lane); return;
        }
    } else if constexpr (MODE != ROWS) {
        switch ((ph.b + 7) / 8) {
            case 2: phase_large<2, RT, MODE>(tile, pitch, w, bases, ph, L, warp, lane); return;
            case 3: phase_large<3, RT, MODE>(tile, pitch, w, bases, ph, L, warp, lane); return;
            case 4: phase_large<4, RT, MODE>(tile, pitch, w, bases, ph, L, warp, lane); return;
            case 5: phase_large<5, RT, MODE>(tile, pitch, w, bases, ph, L, warp, lane); return;
            case 6: phase_large<6, RT, MODE>(tile, pitch, w, bases, ph, L, warp, lane); return;
            case 7: phase_large<7, RT, MODE>(tile, pitch, w, bases, ph, L, warp, lane); return;
            default: phase_large<8, RT, MODE>(tile, pitch, w, bases, ph, L, warp, lane); return;
        }
    }
#undef HARP_F32_CASE
}

// ------------------------------------------------------------------ the pass

// x: batch of n vectors of d coordinates; ROWS, RUNS: vector r at x + r * ld, coordinates contiguous; COLS: coordinate
// i at x + i * ld, vectors contiguous.  sign_at: 0 none, 1 signs on the operands of the pass's first stage (forward), 2 on
// its results (transpose) -- folded into that stage's kernels in shared memory.
template <int RT, int MODE, bool BIG>
__global__ void __launch_bounds__(kF32Threads, 1)
harp_f32_pass_kernel(float *__restrict__ x, int64_t n, int64_t ld, const float *__restrict__ blocks,
                     const int8_t *__restrict__ signs, int transpose, int sign_at, int n_row_tiles, int n_parts, int32_t *err,
                     const __grid_constant__ CUtensorMap tmap, const F32Pass P) {
    constexpr int R = 32 * RT;
    extern __shared__ __align__(16) float smem_raw[];
    float *smem = smem_raw + (((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u) >> 2);       // swizzled boxes start on 1024-byte boundaries
    __shared__ __align__(8) uint64_t full_bar[kMaxBuf];
    __shared__ int dead;
    const int L = P.L, n_c = P.E * L, pitch = P.pitch, n_buf = P.n_buf;
    float *wts = smem + n_buf * P.tile_floats;
    int32_t *tabs = reinterpret_cast<int32_t *>(wts + P.w_floats);   // coordinate of tile index c relative to the group's first, then block bases
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    // Tiles of this CTA: (column group, row tile).  n_parts > 0: the CTA keeps one group and takes every n_parts-th row
    // tile, so that the CTAs of neighbouring groups, whose short runs share DRAM bursts, are at the same rows at the same
    // time; n_parts == 0: an equal share of the group-major list of tiles.
    int cg, rt, n_my, t_step = 1;
    if (n_parts > 0) {
        cg = blockIdx.x % P.n_cg;
        rt = blockIdx.x / P.n_cg;
        t_step = n_parts;
        n_my = rt < n_row_tiles ? (n_row_tiles - rt + n_parts - 1) / n_parts : 0;
    } else {
        const int64_t n_tiles = (int64_t)P.n_cg * n_row_tiles;
        const int64_t per = n_tiles / gridDim.x, extra = n_tiles % gridDim.x;
        const int64_t t0 = blockIdx.x * per + min((int64_t)blockIdx.x, extra);
        n_my = (int)(per + ((int64_t)blockIdx.x < extra ? 1 : 0));
        cg = (int)(t0 / n_row_tiles);
        rt = (int)(t0 - (int64_t)cg * n_row_tiles);
    }
    auto advance = [&](int &c, int &r) {
        r += t_step;
        if (n_parts == 0 && r == n_row_tiles) { r = 0; ++c; }
    };
    auto group_base = [&](int c) {                             // coordinate of tile index 0
        const int hi = c / P.n_lo, lo = c - hi * P.n_lo;
        return (int64_t)hi * P.S * P.E + (int64_t)lo * L;
    };
    auto tile_addr = [&](int c, int r) { return x + (int64_t)r * R * ld + group_base(c); };
    for (int c = threadIdx.x; c < n_c; c += kF32Threads) tabs[c] = (c / L) * (int)P.S + c % L;
    for (int p = 0; p < P.n_ph; ++p) {
        const F32Phase &ph = P.ph[p];
        for (int k = threadIdx.x; k < ph.n_blk; k += kF32Threads) {
            const int l = k % L, rr = k / L, r = rr % ph.ls, a = rr / ph.ls;
            tabs[ph.base_off + k] = (a * ph.b * ph.ls + r) * L + l;
        }
        // columns of padding behind a kernel row: zero once, never written again
        for (int q = threadIdx.x; q < ph.n_blk * ph.b; q += kF32Threads)
            for (int j = ph.b; j < ph.pitch; ++j) wts[ph.w_off + q * ph.pitch + j] = 0.f;
    }
    if (threadIdx.x == 0) {
        for (int b = 0; b < kMaxBuf; ++b) harp_tm::mbar_init(smem_u32(&full_bar[b]), 1);
        dead = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();

    auto load_kernels = [&](int c) {
        const int hi = c / P.n_lo, lo = c - hi * P.n_lo;
        for (int p = 0; p < P.n_ph; ++p) {
            const F32Phase &ph = P.ph[p];
            const int b = ph.b, bb = b * b, ls = ph.ls, hi_blk = hi * (P.E / (b * ls));
            const int64_t s = P.S * ls;
            for (int e = threadIdx.x; e < ph.n_blk * bb; e += kF32Threads) {
                const int k = e / bb, q = e - k * bb, i = q / b, j = q - i * b;
                const int l = k % L, rr = k / L, a = rr / ls, r = rr - a * ls;
                const int64_t blk = (hi_blk + a) * s + (int64_t)r * P.S + (int64_t)lo * L + l;
                cp_async4(wts + ph.w_off + k * b * ph.pitch + (transpose ? j * ph.pitch + i : i * ph.pitch + j), blocks + ph.k_off + blk * bb + q);
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    auto fold_signs = [&](int c) {
        const F32Phase &ph = P.ph[0];
        const int64_t base = group_base(c);
        for (int q = threadIdx.x; q < ph.n_blk * ph.b; q += kF32Threads) {
            const int k = q / ph.b, i = q - k * ph.b;
            if (signs[base + tabs[tabs[ph.base_off + k] + i * ph.ls * L]] >= 0) continue;
            float *kw = wts + ph.w_off + k * ph.b * ph.pitch;
            for (int j = 0; j < ph.b; ++j) {
                float &e = sign_at == 1 ? kw[i * ph.pitch + j] : kw[j * ph.pitch + i];
                e = -e;
            }
        }
    };
    auto stopped = [&] { return *(volatile int *)&dead != 0; };
    // ROWS, COLS: one thread, as few bulk copies as cover the tile (each one costs some 200 cycles to issue), completion on the buffer's mbarrier.  RUNS: every thread its chunks.
    auto copy_in = [&](int c, int r, int b) {
        float *tile = smem + b * P.tile_floats;
        if constexpr (MODE == RUNS) {
            const float *src = tile_addr(c, r);
            const int left = (int)min((int64_t)R, n - (int64_t)r * R);
            for (int row = warp; row < left; row += kWarps)
#pragma unroll 4
                for (int q = 4 * lane; q < n_c; q += 128) cp_async16(tile + row * pitch + q, src + (int64_t)row * ld + tabs[q]);
            asm volatile("cp.async.commit_group;" ::: "memory");
        } else if (threadIdx.x == 0 && !stopped()) {
            const uint32_t bar = smem_u32(&full_bar[b]), dst = smem_u32(tile), box_bytes = 4u * (uint32_t)(n_c / P.n_box * R);
            harp_tm::mbar_expect_tx(bar, box_bytes * (uint32_t)P.n_box);   // past the end of the batch the engine fills zeros
            for (int a = 0; a < P.n_box; ++a) {
                if constexpr (MODE == ROWS) harp_tm::tma_load_3d(dst + a * box_bytes, &tmap, 0, r * R, (int)(group_base(c) >> 5) + a * P.box_e, bar);
                else harp_tm::tma_load_3d(dst + a * box_bytes, &tmap, r * R, (c % P.n_lo) * L, (c / P.n_lo) * P.E + a * P.box_e, bar);
            }
        }
    };
    auto copy_out = [&](int c, int r, int b) {
        const float *tile = smem + b * P.tile_floats;
        if constexpr (MODE == RUNS) {
            float *dst = tile_addr(c, r);
            const int left = (int)min((int64_t)R, n - (int64_t)r * R);
            for (int row = warp; row < left; row += kWarps)
                for (int q0 = 4 * lane; q0 < n_c; q0 += 512) {
                    float4 v[4];
#pragma unroll
                    for (int k = 0; k < 4; ++k)
                        if (q0 + 128 * k < n_c) v[k] = *reinterpret_cast<const float4 *>(tile + row * pitch + q0 + 128 * k);
#pragma unroll
                    for (int k = 0; k < 4; ++k)
                        if (q0 + 128 * k < n_c) *reinterpret_cast<float4 *>(dst + (int64_t)row * ld + tabs[q0 + 128 * k]) = v[k];
                }
        } else if (threadIdx.x == 0 && !stopped()) {
            const uint32_t src = smem_u32(tile), box_bytes = 4u * (uint32_t)(n_c / P.n_box * R);
            for (int a = 0; a < P.n_box; ++a) {
                if constexpr (MODE == ROWS) harp_tm::tma_store_3d(&tmap, 0, r * R, (int)(group_base(c) >> 5) + a * P.box_e, src + a * box_bytes);
                else harp_tm::tma_store_3d(&tmap, r * R, (c % P.n_lo) * L, (c / P.n_lo) * P.E + a * P.box_e, src + a * box_bytes);
            }
            harp_tm::bulk_commit();
        }
    };

    int cur_cg = cg, cg_in = cg, rt_in = rt, buf = 0, buf_in = 0;
    [[maybe_unused]] uint32_t parity = 0;                      // bit b: phase of buffer b's barrier
    if (n_my > 0) load_kernels(cg);
    // plan data only up to here: may run under the kernel before this one
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int ahead = MODE == RUNS ? 1 : n_buf - 1;            // tiles in flight in front of the one being multiplied
    for (int t = 0; t < ahead && t < n_my; ++t) {
        copy_in(cg_in, rt_in, buf_in);
        advance(cg_in, rt_in);
        buf_in = buf_in + 1 == n_buf ? 0 : buf_in + 1;
    }
    for (int t = 0; t < n_my; ++t, advance(cg, rt)) {
        float *tile = smem + buf * P.tile_floats;
        const bool fresh = t == 0 || cg != cur_cg;
        if (cg != cur_cg) {
            cur_cg = cg;
            load_kernels(cg);
        }
        if constexpr (MODE == RUNS) {
            asm volatile("cp.async.wait_all;" ::: "memory");
        } else {
            if (fresh) asm volatile("cp.async.wait_all;" ::: "memory");
            const uint32_t bar = smem_u32(&full_bar[buf]), par = (parity >> buf) & 1u;
            uint32_t it = 0;
            while (!harp_tm::mbar_try(bar, par)) {
                if (++it > kF32Spin || ((it & 63) == 63 && stopped())) {
                    *(volatile int *)&dead = 1;                // from here on nothing is copied any more
                    atomicExch(err, 101);
                    parity ^= 1u << buf;        // (undone below: the phase is still awaited)
                    break;
                }
            }
            parity ^= 1u << buf;
        }
        __syncthreads();
        if (MODE == RUNS && n_buf == 2 && t + 1 < n_my) {      // under the arithmetic of this tile
            copy_in(cg_in, rt_in, buf_in);
            advance(cg_in, rt_in);
            buf_in ^= 1;
        }
        if (fresh && sign_at) {
            fold_signs(cg);
            __syncthreads();
        }
        for (int k = 0; k < P.n_ph; ++k) {
            if (k > 0) __syncthreads();
            const F32Phase &ph = P.ph[transpose ? P.n_ph - 1 - k : k];
            if (!BIG && ph.pair) {
                const F32Phase &lo = ph.pair == 1 ? ph : *(&ph - 1);
                const float *w1 = wts + lo.w_off, *w2 = wts + (&lo + 1)->w_off;
                if constexpr (MODE == ROWS) rm_contig_4x4<RT>(tile, w1, w2, lo.n_blk / 4, transpose, warp, lane);
                else if constexpr (MODE == COLS) col_phase_4x4<RT>(tile, w1, w2, lo, L, transpose, warp, lane);
                ++k;
            } else {
                run_phase<RT, MODE, BIG>(tile, pitch, wts + ph.w_off, tabs + ph.base_off, ph, L, warp, lane);
            }
        }
        if (MODE != RUNS) harp_tm::fence_async_smem();         // results before the copy engine reads them
        __syncthreads();
        copy_out(cg, rt, buf);
        if constexpr (MODE != RUNS) {
            if (t + ahead < n_my) {
                // the buffer of the tile before this one is loaded next: its store must have been read
                if (threadIdx.x == 0) asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");
                copy_in(cg_in, rt_in, buf_in);
                advance(cg_in, rt_in);
                buf_in = buf_in + 1 == n_buf ? 0 : buf_in + 1;
            }
        } else {
            __syncthreads();                                   // the buffer is free for the copy after next
            if (n_buf == 1 && t + 1 < n_my) {
                copy_in(cg_in, rt_in, 0);
                advance(cg_in, rt_in);
            }
        }
        buf = buf + 1 == n_buf ? 0 : buf + 1;
    }
    if (MODE != RUNS && threadIdx.x == 0) {
        harp_tm::bulk_wait0();
        if (stopped()) ring_drain(parity, n_buf, kF32Spin, [&](int k, uint32_t phase) { return harp_tm::mbar_try(smem_u32(&full_bar[k]), phase); });
    }
}

// Fixed permutation and signs of fp32 rows, in place, whole rows through shared memory: out[i] = +-in[table[i]], table: the source of every
// coordinate (the permutation forward, its inverse for the transpose) with the sign in the top bit.  Groups of R rows come by asynchronous 16-byte
// copies, the next one (n_buf = 2) while this one is gathered; an entry of the table is read once for the rows of a group.  harp_permute.h
// says where the pieces of a row lie.
constexpr int kPermuteThreads = 512;
__global__ void __launch_bounds__(kPermuteThreads, 2)
harp_f32_permute_kernel(float *__restrict__ x, int64_t n, int d, int R, int n_buf, const int32_t *__restrict__ table) {
    extern __shared__ __align__(16) float smem[];
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");        // (whoever comes next waits for this grid's end before it touches a row)
    const int pieces = d / 4, pitch = permute_pitch<4>(d);
    const int64_t groups = (n + R - 1) / R;
    auto copy_in = [&](int64_t g, float *buf) {
        if (g < groups) {
            const int rows = (int)min((int64_t)R, n - g * R);
            const float *src = x + g * R * d;
            for (int r = 0; r < rows; ++r)
#pragma unroll 4
                for (int c = threadIdx.x; c < pieces; c += kPermuteThreads) cp_async16(buf + r * pitch + 4 * permute_piece<4>(c), src + (int64_t)r * d + 4 * c);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    asm volatile("griddepcontrol.wait;" ::: "memory");
    copy_in(blockIdx.x, smem);
    int buf = 0;
    for (int64_t g = blockIdx.x; g < groups; g += gridDim.x) {
        if (n_buf == 2) {
            copy_in(g + gridDim.x, smem + (buf ^ 1) * R * pitch);
            asm volatile("cp.async.wait_group 1;" ::: "memory");
        } else {
            asm volatile("cp.async.wait_group 0;" ::: "memory");
        }
        __syncthreads();
        const int rows = (int)min((int64_t)R, n - g * R);
        const float *tile = smem + buf * R * pitch;
        float *dst = x + g * R * d;
        for (int c = threadIdx.x; c < pieces; c += kPermuteThreads) {
            const int4 t = __ldg(reinterpret_cast<const int4 *>(table) + c);
            const int src[4] = {t.x, t.y, t.z, t.w};
            int at[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) at[k] = permute_place<4>(src[k] & 0x7fffffff);
            for (int r = 0; r < rows; ++r) {
                float o[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) o[k] = __uint_as_float(__float_as_uint(tile[r * pitch + at[k]]) ^ ((uint32_t)src[k] & 0x80000000u));
                *reinterpret_cast<float4 *>(dst + (int64_t)r * d + 4 * c) = make_float4(o[0], o[1], o[2], o[3]);
            }
        }
        __syncthreads();                                       // the buffer is free
        if (n_buf == 2) buf ^= 1;
        else copy_in(g + gridDim.x, smem);
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
}

}  // namespace

struct F32Plan {
    int n_pass[2] = {0, 0};            // [0] rows, [1] columns
    F32Pass pass[2][kMaxF32Passes];
    int permute_rows = 0;              // most rows of a group of the permutation kernel (0: identity), its buffers, and tables per direction
    int permute_bufs = 0;
    int32_t *d_table[2] = {nullptr, nullptr};
    int sms = 148;
    int32_t *d_err = nullptr;          // device word, set when a wait gave up
    void *encode = nullptr;            // encoder of tensor maps
};

namespace {

constexpr int64_t kMaxF32Vectors = (int64_t)1 << 30;      // rows or columns of a call: coordinates of a bulk copy are 32-bit

const StageTable &f32_table(const harp_plan *p) { return p->fused.m > 0 && p->d_fused_blocks ? p->fused : p->st; }
const float *f32_blocks(const harp_plan *p) { return p->fused.m > 0 && p->d_fused_blocks ? p->d_fused_blocks : p->d_blocks; }

int kernel_pitch(int b, bool big) {
    if (big && b > 8) return (b + 7) / 8 * 8;
    return b == 2 ? 2 : (b + 3) / 4 * 4;
}

constexpr int kSmemMax = 226 * 1024;

// stages [t0, t1) as one pass with L positions and 32 * RT rows per tile; false if it does not fit.  H > 1 (only from stride 1
// on): the tile takes H neighbouring groups of coordinates
bool make_pass(const StageTable &st, int64_t d, int t0, int t1, int L, int H, int RT, bool col, F32Pass &P) {
    const int64_t S = st.s[t0];
    int64_t E = 1;
    bool big = false;
    for (int t = t0; t < t1; ++t) { E *= st.b[t]; big = big || st.b[t] > 16; }
    if (t1 - t0 > kMaxF32Phases || S % L != 0 || (S > 1 && H > 1) || (d / E) % H != 0) return false;
    E *= H;
    const int64_t n_c = E * L;
    int64_t w = 0;
    const int mode = col ? COLS : S == 1 ? ROWS : RUNS;
    if (mode == ROWS && (big || L != 1 || n_c % 32 != 0)) return false;
    if (mode == RUNS && L % 4 != 0) return false;
    if (n_c > 8192) return false;
    // RUNS: rows an odd number of 16-byte units apart
    const int64_t pitch = mode == RUNS ? n_c + ((n_c / 4) % 2 == 0 ? 4 : 0) : 32 * RT;
    const int64_t tile = mode == RUNS ? 32 * RT * pitch : n_c * pitch;
    // a bulk copy covers at most 256 places (COLS) or 256 runs of 32 coordinates (ROWS)
    const int64_t places = mode == ROWS ? n_c / 32 : E;
    int n_box = 1;
    while (places % n_box != 0 || places / n_box > 256) ++n_box;
    P = F32Pass{};
    P.mode = mode; P.n_box = n_box; P.box_e = (int32_t)(places / n_box); P.pitch = (int32_t)pitch; P.tile_floats = (int32_t)((tile + 3) / 4 * 4);
    P.n_ph = t1 - t0; P.E = (int32_t)E; P.L = L; P.RT = RT; P.S = S; P.d = d; P.big = big;
    P.n_lo = (int32_t)(S / L);
    P.n_cg = (int32_t)(d / n_c);
    for (int t = t0; t < t1; ++t) {
        F32Phase &ph = P.ph[t - t0];
        ph.b = st.b[t];
        ph.ls = (int32_t)(st.s[t] / S);
        ph.n_blk = (int32_t)(n_c / st.b[t]);
        ph.pitch = kernel_pitch(st.b[t], big);
        ph.w_off = (int32_t)w;
        ph.k_off = st.off[t];
        w += (int64_t)ph.n_blk * st.b[t] * ph.pitch;
        w = (w + 3) / 4 * 4;
    }
    P.w_floats = (int32_t)w;
    int64_t tab = n_c;
    for (int p = 0; p < P.n_ph; ++p) { P.ph[p].base_off = (int32_t)tab; tab += P.ph[p].n_blk; }
    for (int p = 0; p + 1 < P.n_ph; ++p)
        if (!big && P.ph[p].pair == 0 && P.ph[p].b == 4 && P.ph[p + 1].b == 4 && (mode == COLS || (mode == ROWS && p == 0))) { P.ph[p].pair = 1; P.ph[p + 1].pair = 2; }
    // a radix above 16 is bound by fetching its block kernels, once for all the rows of a lane: two rows a lane and one buffer
    // beat one row and two (11008 = 256 x 43: half the fetches; the exposed copies are a quarter of a tile's time)
    const int most = mode == RUNS ? 2 : kMaxBuf, least = mode == RUNS && big ? 1 : 2;
    for (P.n_buf = most; P.n_buf >= least; --P.n_buf) {
        const int64_t smem = ((int64_t)P.n_buf * P.tile_floats + w + tab) * 4 + 1024;
        if (smem <= kSmemMax) { P.smem = (int32_t)smem; break; }
    }
    if (P.n_buf < least) return false;
    return true;
}

// A pass of harp_regs.cu or harp_big.cu against one of the kernel above, in trips.  Covers of 5528 batches of rows and 1627 matrices, d = 256 .. 32768,
// against covers without those passes: with 0.75 0.3 % of them more than 4 or 5 % slower, rows on average 0.729 of the time and columns 0.939; with
// 0.5 0.6 %, 0.731 and 0.939, with 0.9 0.3 %, 0.730 and 0.956.
constexpr double kRegCost = 0.75;

// Cost of a pass relative to one trip of the rows through HBM.  What moves it: 16- and 32-byte runs of the row-mode
// copies, one row per lane (every kernel load serves half as much arithmetic), phases with fewer blocks than warps.
double pass_cost(const F32Pass &P, bool col) {
    double c = 1.0, mac = 0.0;
    for (int p = 0; p < P.n_ph; ++p) mac += P.ph[p].b;
    if (!col && P.S > 1) c += P.L == 4 ? 1.0 : P.L == 8 ? 0.1 : 0.0;
    if (P.RT == 1) c += 0.02 * mac;
    if (P.n_buf == 2 && P.mode != RUNS) c += 0.2;
    for (int p = 0; p < P.n_ph; ++p) {
        const int units = P.ph[p].b > 16 ? 2 * P.ph[p].n_blk : P.mode == COLS ? P.ph[p].n_blk / 2 : P.ph[p].n_blk / 4;
        if (units < kWarps) c += 0.2;
    }
    return c;
}

// cheapest cover of the stages by passes (dynamic program over the stage boundaries)
int plan_passes(const StageTable &st, const StageTable &orig, int64_t d, bool col, F32Pass *out) {
    struct Best { double cost; int from; F32Pass pass; int n; };
    std::vector<Best> best((size_t)st.m + 1, Best{1e30, -1, F32Pass{}, 0});
    best[0].cost = 0.0;
    for (int t0 = 0; t0 < st.m; ++t0) {
        if (best[(size_t)t0].cost > 1e29) continue;
        // passes of harp_regs.cu run the plan's own stages (its small radices are fused in st, which rounds their products)
        for (int t1 = t0 + 1; t1 <= st.m; ++t1) {
            auto stage_at = [&](int64_t stride) {
                int o = 0;
                while (o < orig.m && orig.s[o] < stride) ++o;
                return o == orig.m || orig.s[o] == stride ? o : -1;
            };
            const int o0 = stage_at(st.s[t0]), o1 = t1 < st.m ? stage_at(st.s[t1]) : orig.m;
            F32Pass P{};
            if (o0 < 0 || o1 < 0 || o1 - o0 > 11) continue;
            if (!harp_regs_pass(orig, d, o0, o1, col, P.reg) && (col || o1 != o0 + 1 || !harp_big_pass(orig, d, o0, P.reg))) continue;
            const double c = best[(size_t)t0].cost + kRegCost;
            if (c < best[(size_t)t1].cost) best[(size_t)t1] = Best{c, t0, P, best[(size_t)t0].n + 1};
        }
        for (int t1 = t0 + 1; t1 <= st.m; ++t1)
            for (int RT = 1; RT <= 2; ++RT)
                for (int L = 1, H = 1; L <= 32; L *= 2, H = st.s[t0] == 1 ? L : 1) {
                    F32Pass P;
                    if (!make_pass(st, d, t0, t1, st.s[t0] == 1 ? 1 : L, H, RT, col, P)) continue;
                    const double c = best[(size_t)t0].cost + pass_cost(P, col);
                    if (c < best[(size_t)t1].cost) best[(size_t)t1] = Best{c, t0, P, best[(size_t)t0].n + 1};
                }
    }
    const Best &last = best[(size_t)st.m];
    if (last.cost > 1e29 || last.n > kMaxF32Passes) return 0;
    for (int t = st.m, i = last.n - 1; t > 0; t = best[(size_t)t].from, --i) out[i] = best[(size_t)t].pass;
    return last.n;
}

typedef CUresult (*EncodeTiled)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *, const cuuint64_t *,
                                const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle,
                                CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

// row-mode runs below a 128-byte line: see the kernel's tile order (it keeps parts * n_cg of the SMs busy)
int pass_parts(const F32Plan *fp, const F32Pass &P, int64_t n_row_tiles) {
    return P.mode == RUNS && P.L < 32 && P.n_cg <= fp->sms ? (int)std::min<int64_t>(n_row_tiles, fp->sms / P.n_cg) : 0;
}

template <int RT, int MODE, bool BIG>
cudaError_t launch_f32(const F32Plan *fp, const F32Pass &P, float *x, int64_t n, int64_t ld, const float *blocks, const int8_t *signs,
                       int transpose, int sign_at, cudaStream_t stream) {
    auto kern = harp_f32_pass_kernel<RT, MODE, BIG>;
    const cudaError_t ae = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemMax);
    if (ae != cudaSuccess) return ae;
    const int64_t n_row_tiles = (n + 32 * RT - 1) / (32 * RT);
    const int64_t n_tiles = n_row_tiles * P.n_cg;
    const int n_parts = pass_parts(fp, P, n_row_tiles);
    CUtensorMap tmap = {};
    if (MODE != RUNS) {
        const auto enc = reinterpret_cast<EncodeTiled>(fp->encode);
        const cuuint32_t ones[3] = {1, 1, 1};
        CUresult r;
        if (MODE == ROWS) {
            // (coordinate within a run of 32, row, run)
            const cuuint64_t gdim[3] = {32, (cuuint64_t)n, (cuuint64_t)(P.d / 32)}, gstr[2] = {(cuuint64_t)ld * 4, 128};
            const cuuint32_t box[3] = {32, 32 * RT, (cuuint32_t)P.box_e};
            r = enc(&tmap, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, x, gdim, gstr, box, ones, CU_TENSOR_MAP_INTERLEAVE_NONE,
                    CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
        } else {
            // (column, position below the stride, place): the L positions of box_e places
            const cuuint64_t gdim[3] = {(cuuint64_t)n, (cuuint64_t)P.S, (cuuint64_t)(P.d / P.S)}, gstr[2] = {(cuuint64_t)ld * 4, (cuuint64_t)(P.S * ld) * 4};
            const cuuint32_t box[3] = {32 * RT, (cuuint32_t)P.L, (cuuint32_t)P.box_e};
            r = enc(&tmap, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, x, gdim, gstr, box, ones, CU_TENSOR_MAP_INTERLEAVE_NONE,
                    CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
        }
        if (r != CUDA_SUCCESS) return cudaErrorInvalidValue;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(n_parts > 0 ? (int64_t)n_parts * P.n_cg : std::min<int64_t>(n_tiles, fp->sms)));
    cfg.blockDim = dim3(kF32Threads);
    cfg.dynamicSmemBytes = (size_t)P.smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, x, n, ld, blocks, signs, transpose, sign_at, (int)n_row_tiles, n_parts, fp->d_err, tmap, P);
}

template <bool COL>
harp_status_t run_passes(const harp_plan *plan, float *x, int64_t n, int64_t ld, int transpose, cudaStream_t stream) {
    const F32Plan *fp = plan->f32;
    const float *blocks = f32_blocks(plan);
    const int np = fp->n_pass[COL];
    for (int k = 0; k < np; ++k) {
        const int p = transpose ? np - 1 - k : k;
        const F32Pass &P = fp->pass[COL][p];
        // the permutation kernel carries the signs of a permuted plan
        const int sign_at = p == 0 && plan->d_signs && !plan->d_perm ? (transpose ? 2 : 1) : 0;
        cudaError_t err = cudaErrorInvalidValue;
        if (P.reg.shape > 0) {
            err = P.reg.shape > kBigShape ? harp_big_launch(fp->encode, P.reg, fp->sms, x, n, ld, plan->d_blocks, transpose, fp->d_err, stream) : harp_regs_launch(fp->encode, P.reg, fp->sms, x, n, ld, COL ? plan->d_blocks : plan->d_blocks_em, sign_at ? plan->d_signs : nullptr, transpose, fp->d_err, stream);
            g_harp_launches.fetch_add(1, std::memory_order_relaxed);
            if (err != cudaSuccess || cudaGetLastError() != cudaSuccess) return HARP_ERR_CUDA;
            continue;
        }
#define HARP_F32_LAUNCH(M, BIG)                                                                                          \
    err = P.RT == 2 ? launch_f32<2, M, BIG>(fp, P, x, n, ld, blocks, plan->d_signs, transpose, sign_at, stream)          \
                    : launch_f32<1, M, BIG>(fp, P, x, n, ld, blocks, plan->d_signs, transpose, sign_at, stream)
        if constexpr (COL) {
            if (P.big) HARP_F32_LAUNCH(COLS, true);
            else HARP_F32_LAUNCH(COLS, false);
        } else if (P.mode == ROWS) {
            HARP_F32_LAUNCH(ROWS, false);
        } else {
            if (P.big) HARP_F32_LAUNCH(RUNS, true);
            else HARP_F32_LAUNCH(RUNS, false);
        }
#undef HARP_F32_LAUNCH
        g_harp_launches.fetch_add(1, std::memory_order_relaxed);
        if (err != cudaSuccess || cudaGetLastError() != cudaSuccess) return HARP_ERR_CUDA;
    }
    return HARP_OK;
}

harp_status_t permute_rows(const harp_plan *plan, float *x, int64_t n, int transpose, cudaStream_t stream) {
    const F32Plan *fp = plan->f32;
    // two CTAs an SM where two groups' buffers leave room; a small batch is spread over the SMs row by row
    int R = fp->permute_rows;
    while (R > 1 && n < (int64_t)R * 2 * fp->sms) --R;
    const size_t smem = (size_t)fp->permute_bufs * R * permute_pitch<4>(plan->d) * sizeof(float);
    const int per_sm = smem <= 113 * 1024 ? 2 : 1;
    if (cudaFuncSetAttribute(harp_f32_permute_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemMax) != cudaSuccess)
        return HARP_ERR_CUDA;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)std::min<int64_t>((n + R - 1) / R, (int64_t)per_sm * fp->sms));
    cfg.blockDim = dim3(kPermuteThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    const cudaError_t err = cudaLaunchKernelEx(&cfg, harp_f32_permute_kernel, x, n, (int)plan->d, R, fp->permute_bufs, (const int32_t *)fp->d_table[transpose]);
    g_harp_launches.fetch_add(1, std::memory_order_relaxed);
    return err == cudaSuccess && cudaGetLastError() == cudaSuccess ? HARP_OK : HARP_ERR_CUDA;
}

}  // namespace

// Host arrays, an error word and the tables of a permutation: the kernels read the block kernels the plan already keeps.
harp_status_t harp_f32_build(harp_plan *plan) {
    const StageTable &st = f32_table(plan);
    const int64_t d = plan->d;
    if (d > 32768 || !harp_tensor_map_encoder(plan)) return HARP_ERR_UNSUPPORTED;
    for (int t = 0; t < st.m; ++t)
        if (st.b[t] > kMaxF32Radix) return HARP_ERR_UNSUPPORTED;
    F32Plan *fp = new (std::nothrow) F32Plan();
    if (!fp) return HARP_ERR_ALLOC;
    plan->f32 = fp;
    fp->encode = harp_tensor_map_encoder(plan);
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (sms > 0) fp->sms = sms;
    if (cudaMalloc(&fp->d_err, sizeof(int32_t)) != cudaSuccess) return HARP_ERR_ALLOC;
    if (cudaMemset(fp->d_err, 0, sizeof(int32_t)) != cudaSuccess) return HARP_ERR_CUDA;
    if (d % 4 == 0) fp->n_pass[0] = plan_passes(st, plan->st, d, false, fp->pass[0]);
    if (plan->h_perm.empty()) fp->n_pass[1] = plan_passes(st, plan->st, d, true, fp->pass[1]);
    else if (d % 4 == 0) {
        const int64_t row_bytes = permute_pitch<4>(d) * 4;
        fp->permute_bufs = 2 * row_bytes <= kSmemMax ? 2 : 1;
        fp->permute_rows = (int)std::max<int64_t>(1, std::min<int64_t>(4, (112 * 1024) / (fp->permute_bufs * row_bytes)));
        std::vector<int32_t> table[2];
        try {
            for (auto &t : table) t.resize((size_t)d);
        } catch (const std::bad_alloc &) {
            return HARP_ERR_ALLOC;
        }
        for (int64_t i = 0; i < d; ++i) {
            const int32_t from = plan->h_perm[(size_t)i], flip = !plan->h_signs.empty() && plan->h_signs[(size_t)from] < 0 ? INT32_MIN : 0;
            table[0][(size_t)i] = from | flip;
            table[1][(size_t)from] = (int32_t)i | flip;
        }
        for (int k = 0; k < 2; ++k) {
            if (cudaMalloc(&fp->d_table[k], sizeof(int32_t) * (size_t)d) != cudaSuccess) return HARP_ERR_ALLOC;
            if (cudaMemcpy(fp->d_table[k], table[k].data(), sizeof(int32_t) * (size_t)d, cudaMemcpyHostToDevice) != cudaSuccess) return HARP_ERR_CUDA;
        }
    }
    return HARP_OK;
}

void harp_f32_destroy(harp_plan *plan) {
    if (!plan->f32) return;
    if (plan->f32->d_err) cudaFree(plan->f32->d_err);
    for (int32_t *t : plan->f32->d_table)
        if (t) cudaFree(t);
    delete plan->f32;
    plan->f32 = nullptr;
}

const int32_t *harp_f32_source_table(const harp_plan *plan) { return plan->f32 ? plan->f32->d_table[0] : nullptr; }

int32_t harp_f32_error_word(const harp_plan *plan) {
    if (!plan->f32 || !plan->f32->d_err) return 0;
    int32_t v = 0;
    return cudaMemcpy(&v, plan->f32->d_err, sizeof(v), cudaMemcpyDeviceToHost) == cudaSuccess ? v : -1;
}

namespace {

// microseconds of a pass over n vectors, see harp_generic_estimate
double pass_estimate(const F32Plan *fp, const F32Pass &P, int64_t n) {
    if (P.reg.shape > kBigShape) return 6.0 + 2.5e-6 * (double)n * (double)P.reg.d;
    if (P.reg.shape > 0) return 3.2 + 1.3e-6 * (double)n * (double)P.reg.d;
    const int64_t tiles = (n + 32 * P.RT - 1) / (32 * P.RT), n_c = (int64_t)P.E * P.L;
    const int64_t n_parts = pass_parts(fp, P, tiles), per = n_parts > 0 ? (tiles + n_parts - 1) / n_parts : (tiles * P.n_cg + fp->sms - 1) / fp->sms;
    const int64_t groups = n_parts > 0 ? 1 : 1 + (per - 1) / tiles;          // whose block kernels a CTA fetches
    double radices = 0.0;
    for (int k = 0; k < P.n_ph; ++k) radices += P.ph[k].b;
    return 5.1 + 3.3e-4 * (double)(P.w_floats * groups) + 4.06e-4 * (double)(per * n_c * P.RT) * radices + 2.6e-6 * (double)n * (double)P.d;
}

}  // namespace

// Passes by the kernel above cost two or three launches, the block kernels of a column group in every CTA, and tiles of 32 rows; the
// whole-row kernels a wave of CTAs, whatever the batch leaves of it idle: radices (16, 16, 4), whole rows against passes: 128 rows 14 us and
// 25, 256 rows 25 and 25, 512 rows 45 and 28.  The register passes are faster nearly everywhere (d = 8192 in radix 8, whole rows and passes:
// 1 row 23 and 6.6 us, 256 rows 35 and 12, 4096 rows 294 and 104).  One exception, which no time speaks for (42 and 18 us): batches of d = 8192 that
// fill five sixths or more of the whole-row kernel's one wave of tiles of four rows stay with its one launch, to which
// test_small_batches_take_one_launch holds 500 rows.  Smaller batches and other widths take what the estimates say (300 rows of radices
// (4, 3, 4, 2, 4, 4, 7) 55 us whole, 39 in passes; of 2^10, 8 38 and 13).
bool harp_f32_preferred(const harp_plan *plan, int64_t n_rows) {
    const F32Plan *fp = plan->f32;
    if (!fp || fp->n_pass[0] == 0) return false;
    if (plan->opt_f32_passes || harp_generic_supported(plan, HARP_F32) != HARP_OK) return true;
    if (plan->d == 8192 && plan->d_perm == nullptr && harp_generic_max_radix(plan) <= 8 && 6 * n_rows > 20 * fp->sms && n_rows <= 4 * fp->sms) return false;
    double us = 0.0;
    // up to d = 4096 the whole-row CUDA-core kernels of radices up to 8 hold enough rows of a tile to beat passes other than those of harp_regs.cu
    const bool whole = plan->d <= 4096 && harp_generic_max_radix(plan) <= 8;
    for (int p = 0; p < fp->n_pass[0]; ++p) {
        if (whole && fp->pass[0][p].reg.shape == 0) return false;
        us += pass_estimate(fp, fp->pass[0][p], n_rows);
    }
    if (fp->permute_rows) {
        us += 3.5 + 1.3e-6 * (double)n_rows * (double)plan->d;
    }
    // A permutation: where register passes are all there is to choose, the whole-row kernels take more than their estimate (512 rows of d = 4096
    // under a digit reversal 27 us, 1.4 times; 180 batches 0.534 of their time with 1.3, 0.548 with 1); for other plans it holds (256 rows
    // of radices (4, 4, 15, 4) behind a random one 20.7 us, three passes 27.8)
    return us < (fp->permute_rows && whole ? 1.3 : 1.0) * harp_generic_estimate(plan, n_rows, fp->sms);
}

harp_status_t harp_f32_apply(const harp_plan *plan, void *x, int64_t n_rows, harp_dtype_t dtype, int transpose, cudaStream_t stream) {
    const F32Plan *fp = plan->f32;
    if (!fp || dtype != HARP_F32 || fp->n_pass[0] == 0 || n_rows > kMaxF32Vectors || (reinterpret_cast<uintptr_t>(x) & 15u) != 0) return HARP_ERR_UNSUPPORTED;
    float *xf = static_cast<float *>(x);
    harp_status_t rc = HARP_OK;
    if (fp->permute_rows && !transpose) rc = permute_rows(plan, xf, n_rows, 0, stream);
    if (rc == HARP_OK) rc = run_passes<false>(plan, xf, n_rows, plan->d, transpose, stream);
    if (rc == HARP_OK && fp->permute_rows && transpose) rc = permute_rows(plan, xf, n_rows, 1, stream);
    return rc;
}

// Forward apply down the columns of W (dim(plan) x n_cols, row-major, leading dimension ld).
harp_status_t harp_f32_col_apply(const harp_plan *plan, void *W, int64_t n_cols, int64_t ld, harp_dtype_t dtype, cudaStream_t stream) {
    const F32Plan *fp = plan->f32;
    if (!fp || dtype != HARP_F32 || fp->n_pass[1] == 0 || n_cols > kMaxF32Vectors) return HARP_ERR_UNSUPPORTED;
    if ((reinterpret_cast<uintptr_t>(W) & 15u) != 0 || n_cols % 4 != 0 || ld % 4 != 0) return HARP_ERR_UNSUPPORTED;
    // Few columns of a narrow plan with a radix above 8: as rows of the transposed matrix (two transposes, a launch and a trip each) where
    // the whole-row kernel takes them in a wave (369 x 16, radices 41, 3, 3: 27 us, in place 38)
    if (harp_generic_max_radix(plan) > 8 && harp_generic_supported(plan, HARP_F32) == HARP_OK && !plan->opt_f32_passes) {
        double us = 0.0;
        for (int p = 0; p < fp->n_pass[1]; ++p) us += pass_estimate(fp, fp->pass[1][p], n_cols);
        if (us > 2.0 * (3.0 + 2.4e-6 * (double)n_cols * (double)plan->d) + harp_generic_estimate(plan, n_cols, fp->sms)) return HARP_ERR_UNSUPPORTED;
    }
    return run_passes<true>(plan, static_cast<float *>(W), n_cols, ld, 0, stream);
}
