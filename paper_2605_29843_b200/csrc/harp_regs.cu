// fp32 passes over column groups with the block kernels in registers: rows (whole or in runs) and the columns of a matrix.
//
// A pass runs neighbouring stages [t0, t1) on a tile of NC coordinates that is closed under them (see harp_f32.cu, whose passes take every
// other shape).  Its stages are dealt into phases whose radices multiply to at most ten: a thread holds the values of a phase's unit, so that
// up to three stages cost one trip through shared memory, and it keeps the kernels of its units for all tiles that its CTA takes.
// Nothing but values crosses shared memory: a kernel entry that every product of a tile fetches as a broadcast costs as much
// of the shared-memory pipe as the values (the passes of harp_f32.cu: half a wavefront an element and phase of radix 8, here a quarter).
//
// Rows: tiles of G vectors x NC coordinates, eight values of every vector for each of NT threads; NC = 512 where the
// stages and runs of whole 128-byte lines allow (a CTA of two warps waits for less at its barriers, and a small batch spreads
// the block kernels over more SMs).  A vector's tile is 128-byte lines of 32 neighbouring coordinates as the copy engine writes them with its 128-byte swizzle (16-byte piece k
// of line n at k ^ (n mod 8)), which keeps the 32 lanes of a warp on different banks for units in a row (two 16-byte accesses a lane), at stride 8
// and at strides from 32 on; radix-4 units at stride 16 meet two to a bank.
// Columns: tiles of NC = 64 coordinates (80 for units of ten) x 128 columns; a warp owns a unit, a lane four columns.
//
// Tiles come and go by bulk tensor copies over a ring of buffers.  What bounds a pass is HBM: 32 KB in and out take an SM 2.9 k cycles of its share,
// the products of two radix-8 phases 1.1 k.
#include <algorithm>
#include <cstring>
#include <type_traits>

#include "harp_internal.h"
#include "harp_regs.h"
#include "harp_ring.h"
#include "harp_tm_ptx.cuh"

namespace {

using harp_tm::smem_u32;

constexpr int kColThreads = 256;
constexpr int kRegBufs = 6;
constexpr uint32_t kRegSpin = 1u << 22;        // limit of every wait for a bulk copy

// consecutive stages of radices A, B, C (1: none) on units of N values
template <int A_, int B_ = 1, int C_ = 1>
struct Ph {
    static constexpr int A = A_, B = B_, C = C_, N = A * B * C;
    static constexpr int kStages = 1 + (B > 1) + (C > 1);
    static constexpr int kRadices = A + (B > 1 ? B : 0) + (C > 1 ? C : 0);     // kernel entries per value
};
// one stage of radix 16, its units' results shared by four threads: 64 kernel entries and four results each, all values read by each
struct Ph16 { static constexpr int A = 16, B = 1, C = 1, N = 16, kStages = 1, kRadices = 16; };
struct None { static constexpr int A = 1, B = 1, C = 1, N = 1, kStages = 0, kRadices = 0; };

// geometry of a phase: tile stride T, units dealt to U owners, `kSets` each
template <class P, int NC, int T_, int U>
struct Geo {
    static constexpr int T = T_, N = P::N, kUnits = NC / N, kSets = (kUnits + U - 1) / U, V = kSets * N, kW = V * P::kRadices;
    static constexpr bool kAll = kSets * U == kUnits;          // otherwise some owners have no unit
    static __device__ __forceinline__ int unit(int owner, int set) { return kAll ? owner + set * U : min(owner + set * U, kUnits - 1); }
    static __device__ __forceinline__ bool have(int owner) { return kAll || owner < kUnits; }
    // tile coordinate of value i
    static __device__ __forceinline__ int coord(int owner, int i) {
        const int u = unit(owner, i / N);
        return (u / T) * (T * N) + (i % N) * T + u % T;
    }
};

template <int NC, int T_, int U>
struct Geo<Ph16, NC, T_, U> {
    static constexpr int T = T_, N = 16, kUnits = NC / N, kSets = 1, V = 4, kW = 64;
    static_assert(4 * kUnits == U, "four owners a unit");
    static __device__ __forceinline__ int coord(int owner, int i) {
        const int u = owner >> 2;
        return (u / T) * (T * N) + i * T + u % T;
    }
};

// ---- kernels of one stage of radix R, Q values apart, into registers: w[block][i][j] (transposed stage: [j][i]).  A unit's first value is plan
// coordinate `org` + `r`, r below the phase's stride Sp and org a multiple of Sp * N; its blocks are then number org / R + r + b Sp.
// EM: the lanes of a warp own neighbouring blocks and read the element-major copy of the kernels (entry k of block c at k * n_blk + c),
// whole sectors at a time; otherwise they share a block.
template <int R, int Q, int N, bool TR, bool EM>
__device__ __forceinline__ void load_stage(float *w, const float *blocks, int n_blk, int org, int r, int Sp, const int8_t *signs) {
    const float *k0 = blocks + (org / R + r) * (EM ? 1 : R * R);
#pragma unroll
    for (int b = 0; b < N / R; ++b) {
        const float *k = k0 + b * Sp * (EM ? 1 : R * R);
#pragma unroll
        for (int e = 0; e < R * R; e += !EM && R * R % 4 == 0 ? 4 : 1) {
            float q[4];
            if constexpr (EM) {
                q[0] = __ldg(k + e * n_blk);
            } else if constexpr (R * R % 4 == 0) {
                const float4 f = __ldg(reinterpret_cast<const float4 *>(k + e));
                q[0] = f.x; q[1] = f.y; q[2] = f.z; q[3] = f.w;
            } else {
                q[0] = __ldg(k + e);
            }
#pragma unroll
            for (int n = 0; n < (!EM && R * R % 4 == 0 ? 4 : 1); ++n) {
                const int i = (e + n) / R, j = (e + n) % R;
                w[b * R * R + (TR ? j * R + i : i * R + j)] = q[n];
            }
        }
        if (signs) {                                           // the sign diagonal: rows of the first stage's kernels
#pragma unroll
            for (int i = 0; i < R; ++i)
                if (signs[org + r + (b / Q * (Q * R) + b % Q + i * Q) * Sp] < 0) {
#pragma unroll
                    for (int j = 0; j < R; ++j) w[b * R * R + (TR ? j * R + i : i * R + j)] *= -1.f;
                }
        }
    }
}
// pos: plan coordinate of the first value of set n of this owner
template <class P, class G, bool TR, bool EM, typename Pos>
__device__ __forceinline__ void load_phase(float (&w)[G::kW], const float *blocks, const int64_t *off, int d, int Sp, const int8_t *signs, const Pos &pos) {
    if constexpr (std::is_same_v<P, Ph16>) {                   // w[operand][result of this owner's four]
        const int p = pos(0), r = p % Sp, org = p - r, n_blk = d / 16, j0 = 4 * ((int)threadIdx.x & 3);
        const float *k = blocks + off[0] + org / 16 + r;
#pragma unroll
        for (int i = 0; i < 16; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) w[4 * i + j] = __ldg(k + (TR ? (j0 + j) * 16 + i : i * 16 + j0 + j) * n_blk);
        if (signs) {
#pragma unroll
            for (int i = 0; i < 16; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    if (signs[p + (TR ? j0 + j : i) * Sp] < 0) w[4 * i + j] *= -1.f;
        }
        return;
    } else
#pragma unroll
    for (int n = 0; n < G::kSets; ++n) {
        const int p = pos(n), r = p % Sp, org = p - r;
        load_stage<P::A, 1, P::N, TR, EM>(w + n * P::N * P::A, blocks + off[0], d / P::A, org, r, Sp, signs);
        if constexpr (P::B > 1) load_stage<P::B, P::A, P::N, TR, EM>(w + G::V * P::A + n * P::N * P::B, blocks + off[1], d / P::B, org, r, Sp, nullptr);
        if constexpr (P::C > 1) load_stage<P::C, P::A * P::B, P::N, TR, EM>(w + G::V * (P::A + P::B) + n * P::N * P::C, blocks + off[2], d / P::C, org, r, Sp, nullptr);
    }
}

// ---- a stage on the V values of an owner, for M vectors at once
template <int R, int Q, int V, int M>
__device__ __forceinline__ void run_stage(float (&v)[V][M], const float *w) {
#pragma unroll
    for (int b = 0; b < V / R; ++b) {
        const int at = b / Q * (Q * R) + b % Q;
        float y[R][M];
#pragma unroll
        for (int i = 0; i < R; ++i)
#pragma unroll
            for (int j = 0; j < R; ++j)
#pragma unroll
                for (int m = 0; m < M; ++m) y[j][m] = i == 0 ? v[at][m] * w[b * R * R + j] : fmaf(v[at + i * Q][m], w[b * R * R + i * R + j], y[j][m]);
#pragma unroll
        for (int j = 0; j < R; ++j)
#pragma unroll
            for (int m = 0; m < M; ++m) v[at + j * Q][m] = y[j][m];
    }
}
template <class P, class G, bool TR, int M>
__device__ __forceinline__ void run_phase(float (&v)[G::V][M], const float (&w)[G::kW]) {
    auto a = [&] { run_stage<P::A, 1, G::V, M>(v, w); };
    auto b = [&] { if constexpr (P::B > 1) run_stage<P::B, P::A, G::V, M>(v, w + G::V * P::A); };
    auto c = [&] { if constexpr (P::C > 1) run_stage<P::C, P::A * P::B, G::V, M>(v, w + G::V * (P::A + P::B)); };
    if constexpr (!TR) { a(); b(); c(); } else { c(); b(); a(); }
}

__device__ __forceinline__ void lds4(float *v, uint32_t a) {
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]) : "r"(a) : "memory");
}
__device__ __forceinline__ void sts4(uint32_t a, const float *v) {
    asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(a), "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3]) : "memory");
}
__device__ __forceinline__ float lds1(uint32_t a) {
    float v;
    asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ void sts1(uint32_t a, float v) { asm volatile("st.shared.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory"); }

// byte offset of tile coordinate c in a vector's tile (rows).  A unit's first coordinate and the offsets of its other values have no bits in
// common, so place(first + offset) = place(first) ^ place(offset), and the latter is a constant.
__host__ __device__ constexpr uint32_t place(int c) { return (uint32_t)(((c & ~31) | ((((c >> 2) ^ (c >> 5)) & 7) << 2) | (c & 3)) * 4); }

// one phase on the G vectors of a tile of rows, in place
template <class P, class Ge, int G, uint32_t kVec, bool TR>
__device__ __forceinline__ void rows_phase(uint32_t tile, const float (&w)[Ge::kW]) {
    constexpr bool kRun = Ge::T == 1;                          // a unit's values are neighbours
    static_assert(!kRun || Ge::N % 4 == 0, "units in a row move in 16-byte pieces");
    constexpr int U = G < 2 || Ge::V > 8 ? 1 : 2, nA = kRun ? Ge::V / 4 : Ge::V;
    if (!Ge::have(threadIdx.x)) return;
    uint32_t a[nA];
#pragma unroll
    for (int i = 0; i < nA; ++i) {
        const int e = kRun ? 4 * i : i;
        a[i] = tile + (place(Ge::coord(threadIdx.x, e / Ge::N * Ge::N)) ^ place(e % Ge::N * Ge::T));
    }
#pragma unroll
    for (int r = 0; r < G; r += U) {
        float v[U][Ge::V][1];
#pragma unroll
        for (int u = 0; u < U; ++u)
#pragma unroll
            for (int i = 0; i < nA; ++i) {
                if constexpr (kRun) {
                    float q[4];
                    lds4(q, a[i] + (r + u) * kVec);
                    v[u][4 * i][0] = q[0]; v[u][4 * i + 1][0] = q[1]; v[u][4 * i + 2][0] = q[2]; v[u][4 * i + 3][0] = q[3];
                } else {
                    v[u][i][0] = lds1(a[i] + (r + u) * kVec);
                }
            }
#pragma unroll
        for (int u = 0; u < U; ++u) run_phase<P, Ge, TR, 1>(v[u], w);
#pragma unroll
        for (int u = 0; u < U; ++u)
#pragma unroll
            for (int i = 0; i < nA; ++i) {
                if constexpr (kRun) {
                    const float q[4] = {v[u][4 * i][0], v[u][4 * i + 1][0], v[u][4 * i + 2][0], v[u][4 * i + 3][0]};
                    sts4(a[i] + (r + u) * kVec, q);
                } else {
                    sts1(a[i] + (r + u) * kVec, v[u][i][0]);
                }
            }
    }
}

// the same for units shared by four threads: nobody stores before everybody has read
template <class Ge, int G, uint32_t kVec>
__device__ __forceinline__ void rows_phase_shared(uint32_t tile, const float (&w)[Ge::kW]) {
    constexpr bool kRun = Ge::T == 1;
    const uint32_t p0 = place(Ge::coord(threadIdx.x, 0));
    const int j0 = 4 * ((int)threadIdx.x & 3);
    float o[G][4];
#pragma unroll
    for (int r = 0; r < G; ++r) {
        float v[16];
#pragma unroll
        for (int i = 0; i < 16; i += kRun ? 4 : 1) {
            const uint32_t a = tile + (p0 ^ place(i * Ge::T)) + r * kVec;
            if constexpr (kRun) lds4(v + i, a);
            else v[i] = lds1(a);
        }
#pragma unroll
        for (int i = 0; i < 16; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) o[r][j] = i == 0 ? v[0] * w[j] : fmaf(v[i], w[4 * i + j], o[r][j]);
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < G; ++r) {
        if constexpr (kRun) {
            sts4(tile + place(Ge::coord(threadIdx.x, j0)) + r * kVec, o[r]);
        } else {
#pragma unroll
            for (int j = 0; j < 4; ++j) sts1(tile + place(Ge::coord(threadIdx.x, j0 + j)) + r * kVec, o[r][j]);
        }
    }
}

// one phase on a tile of columns, in place: 512 bytes a coordinate, a lane's four columns
template <class P, class Ge, bool TR>
__device__ __forceinline__ void cols_phase(uint32_t tile, const float (&w)[Ge::kW], int warp, int lane) {
    float v[Ge::V][4];
#pragma unroll
    for (int i = 0; i < Ge::V; ++i) lds4(v[i], tile + Ge::coord(warp, i) * 512 + lane * 16);
    run_phase<P, Ge, TR, 4>(v, w);
#pragma unroll
    for (int i = 0; i < Ge::V; ++i) sts4(tile + Ge::coord(warp, i) * 512 + lane * 16, v[i]);
}

// COL false: tiles of G vectors of NC coordinates for NT threads, groups of L neighbouring coordinates (0: NC coordinates in a row); COL true: of 128 columns
template <bool COL_, int NC_, int NT_, int L_, int G_, bool TR_, class P0_, class P1_ = None, class P2_ = None, class P3_ = None>
struct Cfg {
    static constexpr bool COL = COL_, TR = TR_;
    static constexpr int NC = NC_, NT = NT_, L = L_ > 0 ? L_ : 1, G = G_, E = P0_::N * P1_::N * P2_::N * P3_::N;
    static constexpr bool kContig = L_ == 0;
    using P0 = P0_; using P1 = P1_; using P2 = P2_; using P3 = P3_;
    static constexpr int U = COL ? NT / 32 : NT;
    using G0 = Geo<P0, NC, L, U>;
    using G1 = Geo<P1, NC, L * P0::N, U>;
    using G2 = Geo<P2, NC, L * P0::N * P1::N, U>;
    using G3 = Geo<P3, NC, L * P0::N * P1::N * P2::N, U>;
    static_assert(COL_ || NC % 256 == 0, "the swizzle counts lines from multiples of 1024 bytes");
    static constexpr uint32_t kVec = 4u * NC, kTile = COL ? 512u * NC : G * kVec;
    // (six CTAs with fewer buffers each where the kernels leave registers for them: stages (8, 8, 8) and (8), 4096 rows 44.4 -> 50.8 us)
    static constexpr int kPerSm = 256 / NT, kRoom = 196 * 1024 / (kPerSm * (int)kTile), kBufs = kRoom < kRegBufs ? kRoom : kRegBufs;
    static constexpr size_t kSmem = (size_t)kBufs * kTile + 1024;
};

// n_tiles: tiles along the batch; rows: CTA c keeps group c % n_cg and takes every n_parts-th tile; columns: an equal share of the group-major list
template <class C>
__global__ void __launch_bounds__(C::NT, C::kPerSm)
harp_regs_kernel(const float *__restrict__ blocks, const int8_t *__restrict__ signs, int32_t *err, int n_tiles, int n_parts,
                 const __grid_constant__ CUtensorMap tmap, const RegPass P) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ __align__(8) uint64_t full_bar[C::kBufs];
    __shared__ int dead;
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");        // (whoever comes next waits for this grid's end before it touches a row)
    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;           // swizzled boxes start on 1024-byte boundaries
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, owner = C::COL ? warp : threadIdx.x;
    if (threadIdx.x == 0) {
        for (int b = 0; b < C::kBufs; ++b) harp_tm::mbar_init(smem_u32(&full_bar[b]), 1);
        dead = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    int cg, t0, n_my, step = 1;
    if constexpr (!C::COL) {
        cg = blockIdx.x % P.n_cg;
        t0 = blockIdx.x / P.n_cg;
        step = n_parts;
        n_my = t0 < n_tiles ? (n_tiles - t0 + n_parts - 1) / n_parts : 0;
    } else {
        const int64_t all = (int64_t)P.n_cg * n_tiles, per = all / gridDim.x, extra = all % gridDim.x;
        const int64_t first = blockIdx.x * per + min((int64_t)blockIdx.x, extra);
        n_my = (int)(per + ((int64_t)blockIdx.x < extra ? 1 : 0));
        cg = (int)(first / n_tiles);
        t0 = (int)(first - (int64_t)cg * n_tiles);
    }
    float w0[C::G0::kW], w1[C::G1::kW > 0 ? C::G1::kW : 1], w2[C::G2::kW > 0 ? C::G2::kW : 1], w3[C::G3::kW > 0 ? C::G3::kW : 1];
    auto load_kernels = [&](int g) {
        const int hi = g / P.n_lo, lo = g - hi * P.n_lo;
        const int d = (int)P.d, S = (int)P.S;
        // plan coordinate of tile coordinate c; tiles of several short rows (d below NC) repeat the plan, a last group past the end of a row anything
        auto at = [&](int c) {
            if constexpr (C::kContig) return (g * C::NC + c) % d;
            else return hi * S * C::E + c / C::L * S + lo * C::L + c % C::L;
        };
        load_phase<typename C::P0, typename C::G0, C::TR, !C::COL>(w0, blocks, P.off, d, S, signs, [&](int n) { return at(C::G0::coord(owner, n * C::P0::N)); });
        constexpr int s1 = C::P0::kStages, s2 = s1 + C::P1::kStages, s3 = s2 + C::P2::kStages;
        constexpr int m1 = C::P0::N, m2 = m1 * C::P1::N, m3 = m2 * C::P2::N;
        if constexpr (C::P1::kStages > 0) load_phase<typename C::P1, typename C::G1, C::TR, !C::COL>(w1, blocks, P.off + s1, d, S * m1, nullptr, [&](int n) { return at(C::G1::coord(owner, n * C::P1::N)); });
        if constexpr (C::P2::kStages > 0) load_phase<typename C::P2, typename C::G2, C::TR, !C::COL>(w2, blocks, P.off + s2, d, S * m2, nullptr, [&](int n) { return at(C::G2::coord(owner, n * C::P2::N)); });
        if constexpr (C::P3::kStages > 0) load_phase<typename C::P3, typename C::G3, C::TR, !C::COL>(w3, blocks, P.off + s3, d, S * m3, nullptr, [&](int n) { return at(C::G3::coord(owner, n * C::P3::N)); });
    };
    auto stopped = [&] { return *(volatile int *)&dead != 0; };
    auto copy = [&](bool in, int g, int t, int b) {            // thread 0
        const int hi = g / P.n_lo, lo = g - hi * P.n_lo;
        const uint32_t tile = base + b * C::kTile;
        int x0, x1, x2, x3;
        if constexpr (C::COL) { x0 = t * 128; x1 = lo * C::L; x2 = hi * C::E; x3 = 0; }
        else if constexpr (C::kContig) { x0 = 0; x1 = P.linear ? t * (C::G * C::NC / 32) : g * (C::NC / 32); x2 = 0; x3 = P.linear ? 0 : t * C::G; }
        else { x0 = 0; x1 = lo * (C::L / 32); x2 = hi * C::E; x3 = t * C::G; }
        if (in) {
            const uint32_t bar = smem_u32(&full_bar[b]);
            harp_tm::mbar_expect_tx(bar, C::kTile);            // past the ends of the tensor the engine fills zeros
            harp_tm::tma_load_4d(tile, &tmap, x0, x1, x2, x3, bar);
        } else {
            harp_tm::tma_store_4d(&tmap, x0, x1, x2, x3, tile);
            harp_tm::bulk_commit();
        }
    };
    auto advance = [&](int &g, int &t) {
        t += step;
        if (C::COL && t == n_tiles) { t = 0; ++g; }
    };
    int cur = cg, g_in = cg, t_in = t0, buf = 0, buf_in = 0, g = cg, t = t0;
    uint32_t parity = 0;
    if (n_my > 0) load_kernels(cg);
    // plan data only up to here: may run under the kernel before this one
    asm volatile("griddepcontrol.wait;" ::: "memory");
    for (int k = 0; k < C::kBufs - 1 && k < n_my; ++k, ++buf_in, advance(g_in, t_in))
        if (threadIdx.x == 0) copy(true, g_in, t_in, buf_in);
    for (int k = 0; k < n_my; ++k, advance(g, t)) {
        if (C::COL && g != cur) {
            cur = g;
            load_kernels(g);
        }
        const uint32_t tile = base + buf * C::kTile, bar = smem_u32(&full_bar[buf]), par = (parity >> buf) & 1u;
        uint32_t it = 0;
        while (!harp_tm::mbar_try(bar, par)) {
            if (++it > kRegSpin || ((it & 63) == 63 && stopped())) {
                *(volatile int *)&dead = 1;                    // from here on nothing is copied any more
                atomicExch(err, 102);
                parity ^= 1u << buf;                           // (undone below: the phase is still awaited)
                break;
            }
        }
        parity ^= 1u << buf;
        auto phase = [&](auto pi) {
            constexpr int p = decltype(pi)::value;
            using Pp = std::conditional_t<p == 0, typename C::P0, std::conditional_t<p == 1, typename C::P1, std::conditional_t<p == 2, typename C::P2, typename C::P3>>>;
            using Gp = std::conditional_t<p == 0, typename C::G0, std::conditional_t<p == 1, typename C::G1, std::conditional_t<p == 2, typename C::G2, typename C::G3>>>;
            if constexpr (Pp::kStages > 0) {
                const float (&w)[Gp::kW] = [&]() -> const float (&)[Gp::kW] {
                    if constexpr (p == 0) return w0;
                    else if constexpr (p == 1) return w1;
                    else if constexpr (p == 2) return w2;
                    else return w3;
                }();
                if constexpr (C::COL) cols_phase<Pp, Gp, C::TR>(tile, w, warp, lane);
                else if constexpr (std::is_same_v<Pp, Ph16>) rows_phase_shared<Gp, C::G, C::kVec>(tile, w);
                else rows_phase<Pp, Gp, C::G, C::kVec, C::TR>(tile, w);
            }
        };
        constexpr int np = 1 + (C::P1::kStages > 0) + (C::P2::kStages > 0) + (C::P3::kStages > 0);
        using I0 = std::integral_constant<int, C::TR ? np - 1 : 0>;
        phase(I0());
        if constexpr (np > 1) { __syncthreads(); phase(std::integral_constant<int, C::TR ? np - 2 : 1>()); }
        if constexpr (np > 2) { __syncthreads(); phase(std::integral_constant<int, C::TR ? np - 3 : 2>()); }
        if constexpr (np > 3) { __syncthreads(); phase(std::integral_constant<int, C::TR ? np - 4 : 3>()); }
        harp_tm::fence_async_smem();                           // results before the copy engine reads them
        __syncthreads();
        if (threadIdx.x == 0 && !stopped()) {
            copy(false, g, t, buf);
            if (k + C::kBufs - 1 < n_my) {
                // the buffer of the tile before this one is loaded next: its store must have been read
                asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");
                copy(true, g_in, t_in, buf_in);
            }
        }
        if (k + C::kBufs - 1 < n_my) {
            advance(g_in, t_in);
            buf_in = buf_in + 1 == C::kBufs ? 0 : buf_in + 1;
        }
        buf = buf + 1 == C::kBufs ? 0 : buf + 1;
    }
    if (threadIdx.x == 0) {
        harp_tm::bulk_wait0();
        if (stopped()) ring_drain(parity, C::kBufs, kRegSpin, [&](int b, uint32_t phase) { return harp_tm::mbar_try(smem_u32(&full_bar[b]), phase); });
    }
}

typedef CUresult (*EncodeTiled)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *, const cuuint64_t *,
                                const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle,
                                CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

template <class C>
cudaError_t launch(void *encode, const RegPass &P, int sms, float *x, int64_t n, int64_t ld, const float *blocks, const int8_t *signs, int32_t *err, cudaStream_t stream) {
    RegPass Q = P;
    Q.linear = C::kContig && P.d <= C::NC;                     // whole rows: one run of memory, a tile is a piece of it
    CUtensorMap tmap = {};
    cuuint64_t gdim[4], gstr[3];
    cuuint32_t box[4];
    const cuuint32_t ones[4] = {1, 1, 1, 1};
    int64_t n_tiles;
    if (C::COL) {
        // (column, position below the stride, place)
        n_tiles = (n + 127) / 128;
        gdim[0] = (cuuint64_t)n; gdim[1] = (cuuint64_t)P.S; gdim[2] = (cuuint64_t)(P.d / P.S); gdim[3] = 1;
        gstr[0] = (cuuint64_t)ld * 4; gstr[1] = (cuuint64_t)(P.S * ld) * 4; gstr[2] = (cuuint64_t)(P.d * ld) * 4;
        box[0] = 128; box[1] = C::L; box[2] = C::NC / C::L; box[3] = 1;
    } else if (Q.linear) {
        n_tiles = (n * P.d + C::G * C::NC - 1) / (C::G * C::NC);
        gdim[0] = 32; gdim[1] = (cuuint64_t)(n * P.d / 32); gdim[2] = gdim[3] = 1;
        gstr[0] = 128; gstr[1] = gstr[2] = (cuuint64_t)(n * P.d) * 4;
        box[0] = 32; box[1] = C::G * C::NC / 32; box[2] = box[3] = 1;
    } else {
        // (coordinate within a line of 32, line below the stride, place, row)
        const int64_t S = C::kContig ? P.d : P.S;
        n_tiles = (n + C::G - 1) / C::G;
        gdim[0] = 32; gdim[1] = (cuuint64_t)(S / 32); gdim[2] = (cuuint64_t)(P.d / S); gdim[3] = (cuuint64_t)n;
        gstr[0] = 128; gstr[1] = (cuuint64_t)S * 4; gstr[2] = (cuuint64_t)ld * 4;
        box[0] = 32; box[1] = (C::kContig ? C::NC : C::L) / 32; box[2] = C::kContig ? 1 : C::E; box[3] = C::G;
    }
    const auto enc = reinterpret_cast<EncodeTiled>(encode);
    if (enc(&tmap, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, x, gdim, gstr, box, ones, CU_TENSOR_MAP_INTERLEAVE_NONE,
            C::COL ? CU_TENSOR_MAP_SWIZZLE_NONE : CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
        return cudaErrorInvalidValue;
    const auto kern = harp_regs_kernel<C>;
    const cudaError_t ae = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)C::kSmem);
    if (ae != cudaSuccess) return ae;
    const int n_parts = (int)std::max<int64_t>(1, std::min<int64_t>(n_tiles, sms * C::kPerSm / P.n_cg));
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(C::COL ? std::min<int64_t>(n_tiles * P.n_cg, sms) : (int64_t)n_parts * P.n_cg));
    cfg.blockDim = dim3(C::NT);
    cfg.dynamicSmemBytes = C::kSmem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, blocks, signs, err, (int)n_tiles, n_parts, tmap, Q);
}

// ---- the shapes there are kernels for: radices of the pass, coordinates of a tile, run length (0: coordinates in a row)
struct Shape { bool col; int nc, nt, l, n; int b[11]; };
const Shape kShapes[] = {
    {false, 2048, 256, 0, 11, {2, 2, 2, 2, 2, 2, 2, 2, 2, 2, 2}},
    {false, 1024, 128, 0, 10, {2, 2, 2, 2, 2, 2, 2, 2, 2, 2}},
    {false, 512, 64, 0, 9, {2, 2, 2, 2, 2, 2, 2, 2, 2}},
    {false, 512, 64, 0, 8, {2, 2, 2, 2, 2, 2, 2, 2}},
    {false, 512, 64, 0, 3, {8, 8, 8}},
    {false, 512, 64, 0, 3, {4, 4, 4}},
    {false, 512, 128, 0, 2, {16, 16}},
    {false, 512, 64, 64, 1, {8}},
    {false, 512, 64, 32, 2, {8, 2}},
    {false, 2048, 256, 32, 2, {8, 8}},
    {false, 2048, 256, 32, 3, {4, 4, 4}},
    {false, 1792, 256, 32, 2, {8, 7}},
    {false, 1280, 128, 128, 2, {5, 2}},
    {true, 64, kColThreads, 1, 2, {8, 8}},
    {true, 64, kColThreads, 8, 1, {8}},
    {true, 64, kColThreads, 4, 2, {8, 2}},
    {true, 64, kColThreads, 1, 6, {2, 2, 2, 2, 2, 2}},
    {true, 64, kColThreads, 2, 5, {2, 2, 2, 2, 2}},
    {true, 64, kColThreads, 1, 3, {4, 4, 4}},
    {true, 80, kColThreads, 8, 2, {5, 2}},
};
constexpr int kNumShapes = (int)(sizeof(kShapes) / sizeof(kShapes[0]));

}  // namespace

// Stages [t0, t1) of the plan as a pass over rows or columns, if there is a kernel for them.
bool harp_regs_pass(const StageTable &st, int64_t d, int t0, int t1, bool col, RegPass &P) {
    for (int k = 0; k < kNumShapes; ++k) {
        const Shape &sh = kShapes[k];
        if (sh.col != col || sh.n != t1 - t0) continue;
        bool same = true;
        for (int t = t0; t < t1; ++t) same = same && st.b[t] == sh.b[t - t0];
        if (!same) continue;
        const int64_t S = st.s[t0];
        int64_t E = 1;
        for (int t = t0; t < t1; ++t) E *= st.b[t];
        // radix 16 in narrow rows: the whole-row kernels take small batches in one launch
        if (sh.b[0] == 16 && d <= 4096) continue;
        // all of a row's coordinates in a row of memory (whole rows of d up to NC: several to a tile), or runs of L below the stride
        if (sh.l == 0 ? S != 1 || d % 32 != 0 || (d < sh.nc && (sh.nc % d != 0 || E != d)) : S % sh.l != 0) continue;
        P = RegPass{};
        P.shape = k + 1;
        P.S = S;
        P.d = d;
        P.n_lo = sh.l == 0 ? 1 : (int32_t)(S / sh.l);
        P.n_cg = sh.l == 0 ? (int32_t)((d + sh.nc - 1) / sh.nc) : (int32_t)(d / E / sh.l);
        if (sh.l == 0) P.n_lo = P.n_cg;        // (group numbers count along the row)
        for (int t = t0; t < t1; ++t) P.off[t - t0] = st.off[t];
        return col || P.n_cg <= 148;
    }
    return false;
}

cudaError_t harp_regs_launch(void *encode, const RegPass &P, int sms, float *x, int64_t n, int64_t ld, const float *blocks, const int8_t *signs, int transpose,
                             int32_t *err, cudaStream_t stream) {
    const Shape &sh = kShapes[P.shape - 1];
    // vectors of a tile: four where a CTA gets several tiles, fewer for a small batch (more CTAs, each with less to do)
    const int64_t per = n / std::max<int64_t>(1, sms * (256 / sh.nt) / P.n_cg) * (sh.l == 0 && P.d < sh.nc ? P.d : sh.nc) / sh.nc;
    const int G = sh.col ? 1 : per >= 8 ? 4 : per >= 2 ? 2 : 1;
#define HARP_REGS_T(COL, NC, NT, L, G, ...)                                                                                     \
    return transpose ? launch<Cfg<COL, NC, NT, L, G, true, __VA_ARGS__>>(encode, P, sms, x, n, ld, blocks, signs, err, stream)  \
                     : launch<Cfg<COL, NC, NT, L, G, false, __VA_ARGS__>>(encode, P, sms, x, n, ld, blocks, signs, err, stream)
#define HARP_REGS_ROWS(K, NC, NT, L, ...)                                                                                       \
    case K:                                                                                                                     \
        if (G == 4) { HARP_REGS_T(false, NC, NT, L, 4, __VA_ARGS__); }                                                          \
        if (G == 2) { HARP_REGS_T(false, NC, NT, L, 2, __VA_ARGS__); }                                                          \
        HARP_REGS_T(false, NC, NT, L, 1, __VA_ARGS__)
#define HARP_REGS_COLS(K, NC, L, ...)                                                                                           \
    case K: return launch<Cfg<true, NC, kColThreads, L, 1, false, __VA_ARGS__>>(encode, P, sms, x, n, ld, blocks, signs, err, stream)
    using P222 = Ph<2, 2, 2>;
    using P22 = Ph<2, 2>;
    using P8 = Ph<8>;
    using P4 = Ph<4>;
    using P2 = Ph<2>;
    switch (P.shape) {
        HARP_REGS_ROWS(1, 2048, 256, 0, P222, P222, P222, P22);
        HARP_REGS_ROWS(2, 1024, 128, 0, P222, P222, P222, P2);
        HARP_REGS_ROWS(3, 512, 64, 0, P222, P222, P222);
        HARP_REGS_ROWS(4, 512, 64, 0, P222, P222, P22);
        HARP_REGS_ROWS(5, 512, 64, 0, P8, P8, P8);
        HARP_REGS_ROWS(6, 512, 64, 0, P4, P4, P4);
        HARP_REGS_ROWS(7, 512, 128, 0, Ph16, Ph16);
        HARP_REGS_ROWS(8, 512, 64, 64, P8);
        HARP_REGS_ROWS(9, 512, 64, 32, P8, P2);
        HARP_REGS_ROWS(10, 2048, 256, 32, P8, P8);
        HARP_REGS_ROWS(11, 2048, 256, 32, P4, P4, P4);
        HARP_REGS_ROWS(12, 1792, 256, 32, P8, Ph<7>);
        HARP_REGS_ROWS(13, 1280, 128, 128, Ph<5, 2>);
        HARP_REGS_COLS(14, 64, 1, P8, P8);
        HARP_REGS_COLS(15, 64, 8, P8);
        HARP_REGS_COLS(16, 64, 4, P8, P2);
        HARP_REGS_COLS(17, 64, 1, P222, P222);
        HARP_REGS_COLS(18, 64, 2, P222, P22);
        HARP_REGS_COLS(19, 64, 1, P4, P4, P4);
        HARP_REGS_COLS(20, 80, 8, Ph<5, 2>);
        default: return cudaErrorInvalidValue;
    }
#undef HARP_REGS_COLS
#undef HARP_REGS_ROWS
#undef HARP_REGS_T
}
