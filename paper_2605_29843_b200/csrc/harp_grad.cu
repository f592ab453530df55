// Gradient of a scalar loss with respect to the block kernels of a processor (what a fitting
// loop such as Algorithm 3 needs from the apply; the gradient with respect to the rows is the
// transpose apply and needs nothing new).
//
// Forward, rows as row vectors (Algorithm 1):  v_0[i] = s[perm[i]] x[perm[i]],  v_{t+1} = v_t M_t,
// y = v_m.  With G = dL/dy:   g_m = G,   g_t = g_{t+1} M_t^T,
//     dL/dK_t[c][i][j] = sum over rows of  v_t[base_c + i s_t] * g_{t+1}[base_c + j s_t].
//
// The rows are processed in chunks; for a chunk the forward states between steps are kept in global scratch (fp32) and the
// gradient state is walked back step by step.  Every sum over rows is taken in fp64 in a fixed order -- no atomics, so the
// result does not depend on scheduling.
//
// A step is one stage or two: what crosses memory per step is a state forward, and a state, a gradient state and the next
// gradient state backward, so two radix-4 stages (four threads hold sixteen coordinates and transpose 4 x 4 by
// shuffles) or two radix-2 stages (one thread holds four coordinates) in one step halve the traffic that bounds these
// kernels.  Threads own blocks, keep their kernels in registers (read element-major, so that neighbouring threads read
// neighbouring words) and walk over the rows of a slice; the backward kernels write the gradient state and add the
// outer products into fp64 registers in one sweep.  Blocks too large for one thread's registers are shared by threads that
// own some of the results (forward) or some of the rows of the gradient block (backward).  The first step reads x and the
// last dL/dy in their own type.  Radices with no such kernel use the plain one-thread-per-element kernels.
#include <algorithm>
#include <cmath>
#include <type_traits>
#include <map>
#include <mutex>

#include "harp_internal.h"
#include "harp_permute.h"

namespace {

constexpr int kThreads = 256;

// The kernels of one call form a chain, each reading what the one before wrote, and most last
// 5-30 us; they are launched with the programmatic stream-serialisation attribute so that the
// launch of the next one overlaps the tail of the current one.  Each kernel calls
// prior_kernel_done() before it touches anything a kernel before it wrote (griddepcontrol.wait
// returns when that kernel has completed and its writes are visible), and only then lets the
// kernel after it start, so at most one later kernel is resident early.
__device__ __forceinline__ void prior_kernel_done() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// An SM that has to change the split of L1 and shared memory is emptied first, which undoes that overlap and costs a small call more than its
// kernels take.  split: percent of shared memory that every launch asks for, -1: what each kernel needs.
struct Chain { cudaStream_t stream; int split; };

template <typename... KArgs, typename... Args>
void launch_dep(void (*kern)(KArgs...), dim3 grid, dim3 block, size_t smem, const Chain &chain, Args &&...args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = chain.stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributePreferredSharedMemoryCarveout;
    attr[1].val.sharedMemCarveout = (unsigned)std::max(0, chain.split);
    cfg.attrs = attr;
    cfg.numAttrs = chain.split >= 0 ? 2 : 1;
    cudaLaunchKernelEx(&cfg, kern, static_cast<KArgs>(args)...);     // errors are read with cudaGetLastError by the caller
}

template <typename T> __device__ __forceinline__ float to_f32(T v);
template <> __device__ __forceinline__ float to_f32<float>(float v) { return v; }
template <> __device__ __forceinline__ float to_f32<__nv_bfloat16>(__nv_bfloat16 v) { return __bfloat162float(v); }

constexpr int kOwnThreads = 128;   // threads per CTA of the block-owner kernels
constexpr int kFwdRows = 32;       // rows per CTA, forward
constexpr int kSubs = 4;           // backward: warps that share the blocks of a warp and split the rows; their sums are added
                                   // in shared memory, which leaves a quarter of the partial sums to write and read back

// B values s apart; vec: s == 1 and the row is aligned for 16-byte (8-byte bf16) accesses of four
template <int B, typename T> __device__ __forceinline__ void load_block(const T *p, int64_t s, bool vec, float (&v)[B]) {
    if (B % 4 == 0 && vec) {
#pragma unroll
        for (int q = 0; q + 3 < B; q += 4) {
            if constexpr (sizeof(T) == 4) {
                const float4 a = *reinterpret_cast<const float4 *>(p + q);
                v[q] = a.x; v[q + 1] = a.y; v[q + 2] = a.z; v[q + 3] = a.w;
            } else {
                const uint2 a = *reinterpret_cast<const uint2 *>(p + q);
                v[q] = __uint_as_float(a.x << 16); v[q + 1] = __uint_as_float(a.x & 0xffff0000u);
                v[q + 2] = __uint_as_float(a.y << 16); v[q + 3] = __uint_as_float(a.y & 0xffff0000u);
            }
        }
    } else {
#pragma unroll
        for (int i = 0; i < B; ++i) v[i] = to_f32<T>(p[(int64_t)i * s]);
    }
}
template <int B> __device__ __forceinline__ void store_block(float *p, int64_t s, bool vec, const float (&v)[B]) {
    if (B % 4 == 0 && vec) {
#pragma unroll
        for (int q = 0; q + 3 < B; q += 4) *reinterpret_cast<float4 *>(p + q) = make_float4(v[q], v[q + 1], v[q + 2], v[q + 3]);
    } else {
#pragma unroll
        for (int i = 0; i < B; ++i) p[(int64_t)i * s] = v[i];
    }
}
__device__ __forceinline__ float sign_of(const int8_t *signs, int64_t i) { return signs && signs[i] < 0 ? -1.f : 1.f; }

// ---- one stage, forward: out[r][base_c + j s] = sum_i in[r][base_c + i s] K[c][i][j]; a thread owns OUT results of block c
template <int B, int OUT, typename TI>
__global__ void __launch_bounds__(kOwnThreads)
fwd_kernel(const TI *__restrict__ in, const int8_t *__restrict__ signs, int vec, float *__restrict__ out, int64_t rows, int64_t d, int64_t s,
           const float *__restrict__ em) {
    constexpr int PARTS = B / OUT, PER = kOwnThreads / PARTS;
    const int64_t nblk = d / B, c = (int64_t)blockIdx.x * PER + threadIdx.x % PER;
    const int o0 = (threadIdx.x / PER) * OUT;
    if (c >= nblk) return;
    const int64_t alpha = c / s, base = alpha * B * s + (c - alpha * s);
    float k[B][OUT];
#pragma unroll
    for (int i = 0; i < B; ++i) {
        const float sg = sign_of(signs, base + (int64_t)i * s);
#pragma unroll
        for (int j = 0; j < OUT; ++j) k[i][j] = sg * em[(int64_t)(i * B + o0 + j) * nblk + c];
    }
    prior_kernel_done();
    constexpr int U = B >= 8 ? 2 : 4;
    const int64_t r0 = (int64_t)blockIdx.y * kFwdRows, r1 = min(rows, r0 + kFwdRows);
    for (int64_t r = r0; r < r1; r += U) {
        float v[U][B];
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (r + u < r1) load_block<B, TI>(in + (r + u) * d + base, s, vec, v[u]);
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (r + u >= r1) break;
            float o[OUT];
#pragma unroll
            for (int j = 0; j < OUT; ++j) {
                float acc = 0.f;
#pragma unroll
                for (int i = 0; i < B; ++i) acc = fmaf(v[u][i], k[i][j], acc);
                o[j] = acc;
            }
            store_block<OUT>(out + (r + u) * d + base + (int64_t)o0 * s, s, s == 1, o);
        }
    }
}

// CTAs per SM of the backward kernels (registers: 168 per thread from radix 5 to 8, else 128)
constexpr int k44PerSm = 3, kFwd44PerSm = 6;
__host__ __device__ constexpr int bwd_per_sm(int b, int bi, int subs) { return (b >= 5 && b <= 6 ? 12 : 16) / (((b + bi - 1) / bi) * subs); }

// sums of the warps that split the rows, added in the order of the warps; sum k of a lane goes to dst(k)
template <int N, int SUBS, typename Dst>
__device__ __forceinline__ void combine(const double (&acc)[N], double (*sh)[SUBS][32], int sub, int lane, int add, Dst dst) {
    if constexpr (SUBS > 1) {
#pragma unroll
        for (int k = 0; k < N; ++k) sh[k][sub][lane] = acc[k];
        __syncthreads();
#pragma unroll
        for (int k = 0; k < N; ++k)
            if (k % SUBS == sub) {
                double a = sh[k][0][lane];
#pragma unroll
                for (int w = 1; w < SUBS; ++w) a += sh[k][w][lane];
                if (double *p = dst(k)) *p = add ? *p + a : a;
            }
    } else {
#pragma unroll
        for (int k = 0; k < N; ++k)
            if (double *p = dst(k)) *p = add ? *p + acc[k] : acc[k];
    }
}

// ---- one stage, backward: g_out[r][base_c + i s] = sum_j g[r][base_c + j s] K[c][i][j] (when g_out is given) and
// part[slice][i B + j][c] = sum over the slice's rows of v[..i..] g[..j..]; a thread owns BI values of i of block c
template <int B, int BI, int SUBS, typename TV, typename TG>
__global__ void __launch_bounds__(32 * ((B + BI - 1) / BI) * SUBS, bwd_per_sm(B, BI, SUBS))
bwd_kernel(const TV *__restrict__ v, const int8_t *__restrict__ signs, int vec_v, const TG *__restrict__ g, int vec_g, float *__restrict__ g_out,
           int64_t rows, int64_t d, int64_t s, int slice, int add, const float *__restrict__ em, double *__restrict__ part) {
    constexpr int PARTS = (B + BI - 1) / BI;
    __shared__ double sh[SUBS > 1 ? PARTS : 1][SUBS > 1 ? BI * B : 1][SUBS][32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, pt = w / SUBS, sub = w - pt * SUBS, i0 = pt * BI;
    const int64_t nblk = d / B, cc = (int64_t)blockIdx.x * 32 + lane;
    const bool have = cc < nblk;
    const int64_t c = have ? cc : nblk - 1;
    const int64_t alpha = c / s, base = alpha * B * s + (c - alpha * s);
    float k[BI][B], sg[BI];
    double acc[BI * B];
#pragma unroll
    for (int i = 0; i < BI; ++i) {
        sg[i] = i0 + i < B ? sign_of(signs, base + (int64_t)(i0 + i) * s) : 0.f;
#pragma unroll
        for (int j = 0; j < B; ++j) {
            k[i][j] = i0 + i < B ? em[(int64_t)((i0 + i) * B + j) * nblk + c] : 0.f;
            acc[i * B + j] = 0.0;
        }
    }
    prior_kernel_done();
    const int64_t r0 = (int64_t)blockIdx.y * slice, r1 = min(rows, r0 + slice);
    constexpr bool kWhole = B % BI == 0;
    const bool vec_o = s == 1 && kWhole;
#pragma unroll (B >= 7 ? 1 : B <= 3 ? 4 : 2)
    for (int64_t r = r0 + sub; r < r1; r += SUBS) {
        float vv[BI], gg[B];
        if constexpr (kWhole) {
            load_block<BI, TV>(v + r * d + base + (int64_t)i0 * s, s, vec_v, vv);
        } else {
#pragma unroll
            for (int i = 0; i < BI; ++i) vv[i] = i0 + i < B ? to_f32<TV>(v[r * d + base + (int64_t)(i0 + i) * s]) : 0.f;
        }
        load_block<B, TG>(g + r * d + base, s, vec_g, gg);
        double gd[B];
#pragma unroll
        for (int j = 0; j < B; ++j) gd[j] = (double)gg[j];
#pragma unroll
        for (int i = 0; i < BI; ++i) {
            const double vd = (double)(sg[i] * vv[i]);
#pragma unroll
            for (int j = 0; j < B; ++j) acc[i * B + j] += vd * gd[j];
        }
        if (g_out && have) {
            float o[BI];
#pragma unroll
            for (int i = 0; i < BI; ++i) {
                float a = 0.f;
#pragma unroll
                for (int j = 0; j < B; ++j) a = fmaf(gg[j], k[i][j], a);
                o[i] = a;
            }
            float *dst = g_out + r * d + base + (int64_t)i0 * s;
            if constexpr (kWhole) {
                store_block<BI>(dst, s, vec_o, o);
            } else {
#pragma unroll
                for (int i = 0; i < BI; ++i)
                    if (i0 + i < B) dst[(int64_t)i * s] = o[i];
            }
        }
    }
    double *dst = part + (int64_t)blockIdx.y * (B * B) * nblk + c;
    combine<BI * B, SUBS>(acc, SUBS > 1 ? sh[pt] : nullptr, sub, lane, add, [&](int e) -> double * {
        const int ij = i0 * B + e;
        return have && ij < B * B ? dst + (int64_t)ij * nblk : nullptr;
    });
}

// ---- two radix-4 stages of strides s and 4 s.  A unit is sixteen coordinates base + (i1 + 4 i2) s; its four threads q hold,
// in the first stage's order, block i2 = q (coordinates base + 4 q s + i s) and, in the second stage's, block i1 = q
// (base + q s + 4 j s).  S1 (s == 1): the threads of a unit are neighbouring lanes, a row's sixteen values are loaded as
// four 16-byte pieces; otherwise eight neighbouring units share a quarter-warp each, so that accesses are whole sectors.
template <bool S1>
struct Pair44 {
    int q;
    int64_t base, c1, c2;              // first coordinate; block numbers of this thread's two blocks
    bool have;
    __device__ __forceinline__ Pair44(int64_t d, int64_t s, int64_t first_unit) {
        const int lane = threadIdx.x & 31;
        q = S1 ? lane & 3 : lane >> 3;
        const int64_t u = first_unit + (S1 ? lane >> 2 : lane & 7);
        have = u < d / 16;
        const int64_t uu = have ? u : S1 ? 0 : min((int64_t)(lane & 7), d / 16 - 1), alpha = uu / s, beta = uu - alpha * s;     // past the end: any units, neighbours too
        base = alpha * 16 * s + beta;
        c1 = (4 * alpha + q) * s + beta;
        c2 = alpha * 4 * s + beta + q * s;
    }
    // x[i] of thread q becomes x[q] of thread i, by way of kSwap words of the warp's own (a 16-byte store and four loads, free of bank
    // conflicts; two rounds of shuffles and selects are twenty instructions).  The warp synchronises before the words are written again.
    static constexpr int kSwap = 160;
    __device__ __forceinline__ void transpose(float *words, float (&x)[4]) const {
        const int lane = threadIdx.x & 31;
        float *w = words + (S1 ? lane >> 2 : lane & 7) * 20;
        *reinterpret_cast<float4 *>(w + 4 * q) = make_float4(x[0], x[1], x[2], x[3]);
        __syncwarp();
#pragma unroll
        for (int i = 0; i < 4; ++i) x[i] = w[4 * i + q];
    }
};
__device__ __forceinline__ void mul4(const float (&x)[4], const float (&k)[4][4], float (&y)[4]) {        // y_j = sum_i x_i k[i][j]
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        float a = 0.f;
#pragma unroll
        for (int i = 0; i < 4; ++i) a = fmaf(x[i], k[i][j], a);
        y[j] = a;
    }
}
__device__ __forceinline__ void mul4t(const float (&x)[4], const float (&k)[4][4], float (&y)[4]) {       // y_i = sum_j x_j k[i][j]
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        float a = 0.f;
#pragma unroll
        for (int j = 0; j < 4; ++j) a = fmaf(x[j], k[i][j], a);
        y[i] = a;
    }
}

// Rows on their way to the lanes of a Pair44.  A row's coordinates of a warp come by asynchronous copies of 8 or 16 bytes a lane into a
// ring of the warp's own in shared memory, several rows ahead of the one being multiplied: a step reads little per row and thread (16
// bytes a state), so that with loads one row ahead the rows in flight, 12 KB an SM, bounded it at 1.8 TB/s.  S1: a unit's sixteen values
// in a row, 20 words apart in fp32 (both orders of reading then hit 32 banks); otherwise sixteen runs of the eight neighbouring units, four runs and 32 bytes of padding.
template <bool S1, typename T>
struct Rows44 {
    static constexpr int kBytes = sizeof(T) == 2 ? 256 : 640;
    static __device__ __forceinline__ void issue(unsigned char *dst, const T *row, const Pair44<S1> &u, int64_t s) {
        const int lane = threadIdx.x & 31;
        uint32_t to = (uint32_t)__cvta_generic_to_shared(dst);
        if constexpr (S1) {
            const T *src = row + u.base + 4 * u.q;
            if constexpr (sizeof(T) == 2) asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(to + 8 * lane), "l"(src) : "memory");
            else asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(to + (lane >> 2) * 80 + u.q * 16), "l"(src) : "memory");
        } else if constexpr (sizeof(T) == 2) {
            const T *src = row + (u.base - (lane & 7)) + (lane & 15) * s;
            if (lane < 16) asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(to + 16 * lane), "l"(src) : "memory");
        } else {
            const int run = lane >> 1;
            const T *src = row + (u.base - (lane & 7)) + run * s + (lane & 1) * 4;
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(to + 16 * lane + (run >> 2) * 32), "l"(src) : "memory");
        }
    }
    // first stage's order: coordinates base + (4 q + i) s
    static __device__ __forceinline__ void first(const unsigned char *from, const Pair44<S1> &u, float (&v)[4]) {
        const int lane = threadIdx.x & 31;
        if constexpr (S1) load_block<4, T>(reinterpret_cast<const T *>(from + (sizeof(T) == 2 ? 8 * lane : (lane >> 2) * 80 + u.q * 16)), 1, true, v);
        else if constexpr (sizeof(T) == 2) load_block<4, T>(reinterpret_cast<const T *>(from) + 32 * u.q + (lane & 7), 8, false, v);
        else load_block<4, T>(reinterpret_cast<const T *>(from) + 40 * u.q + (lane & 7), 8, false, v);
    }
    // second stage's: base + (q + 4 j) s
    static __device__ __forceinline__ void second(const unsigned char *from, const Pair44<S1> &u, float (&v)[4]) {
        const int lane = threadIdx.x & 31;
        if constexpr (S1) load_block<4, T>(reinterpret_cast<const T *>(from + (lane >> 2) * (sizeof(T) == 2 ? 32 : 80)) + u.q, 4, false, v);
        else if constexpr (sizeof(T) == 2) load_block<4, T>(reinterpret_cast<const T *>(from) + 8 * u.q + (lane & 7), 32, false, v);
        else load_block<4, T>(reinterpret_cast<const T *>(from) + 8 * u.q + (lane & 7), 40, false, v);
    }
};
constexpr int kRing = 8;               // rows in a warp's ring
__device__ __forceinline__ void ring_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
// the oldest row of the ring has arrived, for the whole warp
__device__ __forceinline__ void ring_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(kRing - 1) : "memory");
    __syncwarp();
}

// RING: rows by asynchronous copies (16-byte boundaries: see ring44)
template <bool S1, bool RING, typename TI>
__global__ void __launch_bounds__(kOwnThreads, kFwd44PerSm)
fwd44_kernel(const TI *__restrict__ in, const int8_t *__restrict__ signs, int vec, float *__restrict__ out, int64_t rows, int64_t d, int64_t s, int slice,
             const float *__restrict__ em1, const float *__restrict__ em2) {
    using Rows = Rows44<S1, TI>;
    __shared__ __align__(16) unsigned char ring[RING ? kOwnThreads / 32 : 1][RING ? kRing : 1][RING ? Rows::kBytes : 16];
    __shared__ __align__(16) float words[kOwnThreads / 32][S1 ? 2 : 1][Pair44<S1>::kSwap];
    const int w = threadIdx.x >> 5;
    const Pair44<S1> u(d, s, ((int64_t)blockIdx.x * (kOwnThreads / 32) + w) * 8);
    const int64_t nblk = d / 4, in0 = u.base + 4 * u.q * s, out0 = S1 ? in0 : u.base + u.q * s, os = S1 ? 1 : 4 * s;
    float k1[4][4], k2[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const float sg = sign_of(signs, in0 + i * s);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            k1[i][j] = sg * em1[(int64_t)(i * 4 + j) * nblk + u.c1];
            k2[i][j] = em2[(int64_t)(i * 4 + j) * nblk + u.c2];
        }
    }
    prior_kernel_done();
    const int64_t r0 = (int64_t)blockIdx.y * slice, r1 = min(rows, r0 + slice);
    float *to = out + r0 * d + out0;
    auto row = [&](const float (&x)[4]) {
        float y[4], z[4];
        mul4(x, k1, y);
        u.transpose(words[w][0], y);
        mul4(y, k2, z);
        if (S1) u.transpose(words[w][S1 ? 1 : 0], z);
        if (u.have) store_block<4>(to, os, S1, z);
        to += d;
        if (!RING) __syncwarp();
    };
    if constexpr (RING) {
        const TI *src = in + r0 * d;
#pragma unroll 1
        for (int k = 0; k < kRing; ++k, src += d) {
            if (r0 + k < r1) Rows::issue(ring[w][k], src, u, s);
            ring_commit();
        }
        for (int64_t r = r0; r < r1; ++r, src += d) {
            unsigned char *slot = ring[w][(int)(r - r0) & (kRing - 1)];
            float x[4];
            ring_wait();
            Rows::first(slot, u, x);
            __syncwarp();
            if (r + kRing < r1) Rows::issue(slot, src, u, s);
            ring_commit();
            row(x);
        }
    } else {
        const TI *p = in + r0 * d + in0;
        float x[4][4];
        for (int64_t r = r0; r < r1; r += 4, p += 4 * d) {
#pragma unroll
            for (int n = 0; n < 4; ++n)
                if (r + n < r1) load_block<4, TI>(p + n * d, s, vec, x[n]);
#pragma unroll
            for (int n = 0; n < 4; ++n)
                if (r + n < r1) row(x[n]);
        }
    }
}

template <bool S1, bool RING, typename TV, typename TG>
__global__ void __launch_bounds__(32 * kSubs, k44PerSm)
bwd44_kernel(const TV *__restrict__ v, const int8_t *__restrict__ signs, int vec_v, const TG *__restrict__ g, int vec_g, float *__restrict__ g_out,
             int64_t rows, int64_t d, int64_t s, int slice, int add, const float *__restrict__ em1, const float *__restrict__ em2, double *__restrict__ part1,
             double *__restrict__ part2) {
    using RowsV = Rows44<S1, TV>;
    using RowsG = Rows44<S1, TG>;
    constexpr int kSums = 32 * kSubs * 32 * 8, kRings = kSubs * kRing * (RowsV::kBytes + RowsG::kBytes);
    __shared__ __align__(16) unsigned char smem[RING && kRings > kSums ? kRings : kSums];        // the rings, then the warps' sums
    __shared__ __align__(16) float words[kSubs][2][Pair44<S1>::kSwap];
    const int lane = threadIdx.x & 31, sub = threadIdx.x >> 5;
    const Pair44<S1> u(d, s, (int64_t)blockIdx.x * 8);
    const int64_t nblk = d / 4, first = u.base + 4 * u.q * s, second = S1 ? first : u.base + u.q * s, gs = S1 ? 1 : 4 * s;
    float k1[4][4], k2[4][4], sg[4];           // k1 with the signs of the step's coordinates
    double acc[32];                            // first stage's sums, second stage's
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        sg[i] = sign_of(signs, first + i * s);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            k1[i][j] = sg[i] * em1[(int64_t)(i * 4 + j) * nblk + u.c1];
            k2[i][j] = em2[(int64_t)(i * 4 + j) * nblk + u.c2];
            acc[i * 4 + j] = acc[16 + i * 4 + j] = 0.0;
        }
    }
    prior_kernel_done();
    const int64_t r0 = (int64_t)blockIdx.y * slice + sub, r1 = min(rows, (int64_t)(blockIdx.y + 1) * slice);
    float *w = g_out ? g_out + r0 * d + first : nullptr;
    // x: first stage's order, gy: second stage's
    auto row = [&](const float (&x)[4], const float (&gy)[4]) {
        float y[4], h[4];
        mul4(x, k1, y);
        mul4t(gy, k2, h);
        u.transpose(words[sub][0], y);
        u.transpose(words[sub][1], h);
        {
            double gd[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) gd[j] = (double)gy[j];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const double vd = (double)y[i];
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[16 + i * 4 + j] += vd * gd[j];
            }
        }
        {
            double gd[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) gd[j] = (double)h[j];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const double vd = (double)x[i];
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[i * 4 + j] += vd * gd[j];
            }
        }
        if (w) {                               // (a step with signs is the first one and has no gradient state behind it)
            float o[4];
            mul4t(h, k1, o);
            if (u.have) store_block<4>(w, s, S1, o);
            w += kSubs * d;
        }
    };
    if constexpr (RING) {
        unsigned char *ring_v = smem + sub * kRing * RowsV::kBytes, *ring_g = smem + kSubs * kRing * RowsV::kBytes + sub * kRing * RowsG::kBytes;
        const TV *pv = v + r0 * d;
        const TG *pg = g + r0 * d;
#pragma unroll 1
        for (int k = 0; k < kRing; ++k, pv += kSubs * d, pg += kSubs * d) {
            if (r0 + k * kSubs < r1) {
                RowsV::issue(ring_v + k * RowsV::kBytes, pv, u, s);
                RowsG::issue(ring_g + k * RowsG::kBytes, pg, u, s);
            }
            ring_commit();
        }
        int k = 0;
        for (int64_t r = r0; r < r1; r += kSubs, pv += kSubs * d, pg += kSubs * d, k = (k + 1) & (kRing - 1)) {
            float x[4], gy[4];
            ring_wait();
            RowsV::first(ring_v + k * RowsV::kBytes, u, x);
            RowsG::second(ring_g + k * RowsG::kBytes, u, gy);
            __syncwarp();
            if (r + kRing * kSubs < r1) {
                RowsV::issue(ring_v + k * RowsV::kBytes, pv, u, s);
                RowsG::issue(ring_g + k * RowsG::kBytes, pg, u, s);
            }
            ring_commit();
            row(x, gy);
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncthreads();
    } else {
        const TV *pv = v + r0 * d + first;
        const TG *pg = g + r0 * d + second;
        float nv[4], ng[4];
        if (r0 < r1) {
            load_block<4, TV>(pv, s, vec_v, nv);
            load_block<4, TG>(pg, gs, vec_g, ng);
        }
        for (int64_t r = r0; r < r1; r += kSubs) {
            float x[4], gy[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) { x[i] = nv[i]; gy[i] = ng[i]; }
            pv += kSubs * d;
            pg += kSubs * d;
            if (r + kSubs < r1) {              // the next row's values are on their way
                load_block<4, TV>(pv, s, vec_v, nv);
                load_block<4, TG>(pg, gs, vec_g, ng);
            }
            if (S1) {
                u.transpose(words[sub][0], gy);
                __syncwarp();
            }
            row(x, gy);
            __syncwarp();
        }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i * 4 + j] = sg[i] < 0.f ? -acc[i * 4 + j] : acc[i * 4 + j];
    double *d1 = part1 + (int64_t)blockIdx.y * 16 * nblk + u.c1, *d2 = part2 + (int64_t)blockIdx.y * 16 * nblk + u.c2;
    combine<32, kSubs>(acc, reinterpret_cast<double (*)[kSubs][32]>(smem), sub, lane, add, [&](int e) -> double * {
        return !u.have ? nullptr : e < 16 ? d1 + (int64_t)e * nblk : d2 + (int64_t)(e - 16) * nblk;
    });
}

// ---- four radix-2 stages of strides s, 2 s, 4 s and 8 s (NS = 3: the first three of them) on the same units: a thread holds two stages' blocks in the first order (coordinate
// i of four: pairs i, i ^ 1, then i, i ^ 2) and the other two stages' in the second.  As much register space for kernels and sums as two
// radix-4 stages, and half the state traffic of two radix-2 stages a step.
template <bool S1>
struct Quad2222 : Pair44<S1> {
    int64_t c[4][2];                   // block numbers of this thread: stage, block
    __device__ __forceinline__ Quad2222(int64_t d, int64_t s, int64_t first_unit) : Pair44<S1>(d, s, first_unit) {
        const int64_t alpha = this->base / (16 * s), beta = this->base - alpha * 16 * s;
        const int q = this->q;
#pragma unroll
        for (int b = 0; b < 2; ++b) {
            c[0][b] = (8 * alpha + 2 * q + b) * s + beta;
            c[1][b] = (4 * alpha + q) * 2 * s + b * s + beta;
            c[2][b] = (2 * alpha + b) * 4 * s + q * s + beta;
            c[3][b] = 8 * alpha * s + (q + 4 * b) * s + beta;
        }
    }
};
// stage of pairs (0, 1), (2, 3) (HI = 0) or (0, 2), (1, 3) (HI = 1) with kernels k[block][i][j]; T: transposed kernels
template <int HI, bool T>
__device__ __forceinline__ void mul22(const float (&x)[4], const float (&k)[2][2][2], float (&y)[4]) {
#pragma unroll
    for (int b = 0; b < 2; ++b)
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const int at0 = HI ? b : 2 * b, st = HI ? 2 : 1;
            y[at0 + j * st] = fmaf(x[at0 + st], T ? k[b][j][1] : k[b][1][j], fmaf(x[at0], T ? k[b][j][0] : k[b][0][j], 0.f));
        }
}
template <int HI>
__device__ __forceinline__ void outer22(const double (&x)[4], const double (&g)[4], double *acc) {
#pragma unroll
    for (int b = 0; b < 2; ++b)
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                const int at0 = HI ? b : 2 * b, st = HI ? 2 : 1;
                acc[b * 4 + i * 2 + j] += x[at0 + i * st] * g[at0 + j * st];
            }
}
__device__ __forceinline__ void widen(const float (&x)[4], double (&y)[4]) {
#pragma unroll
    for (int i = 0; i < 4; ++i) y[i] = (double)x[i];
}
struct Blocks4 { const float *em[4]; };
struct Sums4 { double *part[4]; };

template <int NS, bool S1, typename TI>
__global__ void __launch_bounds__(kOwnThreads, kFwd44PerSm)
fwd2222_kernel(const TI *__restrict__ in, const int8_t *__restrict__ signs, float *__restrict__ out, int64_t rows, int64_t d, int64_t s, int slice, const Blocks4 em) {
    using Rows = Rows44<S1, TI>;
    __shared__ __align__(16) unsigned char ring[kOwnThreads / 32][kRing][Rows::kBytes];
    __shared__ __align__(16) float words[kOwnThreads / 32][S1 ? 2 : 1][Pair44<S1>::kSwap];
    const int w = threadIdx.x >> 5;
    const Quad2222<S1> u(d, s, ((int64_t)blockIdx.x * (kOwnThreads / 32) + w) * 8);
    const int64_t nblk = d / 2, in0 = u.base + 4 * u.q * s, out0 = S1 ? in0 : u.base + u.q * s, os = S1 ? 1 : 4 * s;
    float k[NS][2][2][2];
#pragma unroll
    for (int t = 0; t < NS; ++t)
#pragma unroll
        for (int b = 0; b < 2; ++b)
#pragma unroll
            for (int ij = 0; ij < 4; ++ij)
                k[t][b][ij >> 1][ij & 1] = (t == 0 ? sign_of(signs, in0 + (2 * b + (ij >> 1)) * s) : 1.f) * em.em[t][(int64_t)ij * nblk + u.c[t][b]];
    prior_kernel_done();
    const int64_t r0 = (int64_t)blockIdx.y * slice, r1 = min(rows, r0 + slice);
    const TI *src = in + r0 * d;
    float *to = out + r0 * d + out0;
#pragma unroll 1
    for (int n = 0; n < kRing; ++n, src += d) {
        if (r0 + n < r1) Rows::issue(ring[w][n], src, u, s);
        ring_commit();
    }
    for (int64_t r = r0; r < r1; ++r, src += d, to += d) {
        unsigned char *slot = ring[w][(int)(r - r0) & (kRing - 1)];
        float x[4], y[4];
        ring_wait();
        Rows::first(slot, u, x);
        __syncwarp();
        if (r + kRing < r1) Rows::issue(slot, src, u, s);
        ring_commit();
        mul22<0, false>(x, k[0], y);
        mul22<1, false>(y, k[1], x);
        u.transpose(words[w][0], x);
        mul22<0, false>(x, k[2], y);
        if constexpr (NS == 4) {
            mul22<1, false>(y, k[3], x);
        } else {
#pragma unroll
            for (int i = 0; i < 4; ++i) x[i] = y[i];
        }
        if (S1) u.transpose(words[w][S1 ? 1 : 0], x);
        if (u.have) store_block<4>(to, os, S1, x);
    }
}

template <int NS, bool S1, typename TV, typename TG>
__global__ void __launch_bounds__(32 * kSubs, k44PerSm)
bwd2222_kernel(const TV *__restrict__ v, const int8_t *__restrict__ signs, const TG *__restrict__ g, float *__restrict__ g_out, int64_t rows, int64_t d, int64_t s,
               int slice, int add, const Blocks4 em, const Sums4 part) {
    using RowsV = Rows44<S1, TV>;
    using RowsG = Rows44<S1, TG>;
    constexpr int kSums = 8 * NS * kSubs * 32 * 8, kRings = kSubs * kRing * (RowsV::kBytes + RowsG::kBytes);
    __shared__ __align__(16) unsigned char smem[kRings > kSums ? kRings : kSums];               // the rings, then the warps' sums
    __shared__ __align__(16) float words[kSubs][2][Pair44<S1>::kSwap];
    const int lane = threadIdx.x & 31, sub = threadIdx.x >> 5;
    const Quad2222<S1> u(d, s, (int64_t)blockIdx.x * 8);
    const int64_t nblk = d / 2, first = u.base + 4 * u.q * s;
    float k[NS][2][2][2], sg[4];                // k[0] with the signs of the step's coordinates
    double acc[8 * NS];                        // [stage][block][i][j]
#pragma unroll
    for (int i = 0; i < 4; ++i) sg[i] = sign_of(signs, first + i * s);
#pragma unroll
    for (int t = 0; t < NS; ++t)
#pragma unroll
        for (int b = 0; b < 2; ++b)
#pragma unroll
            for (int ij = 0; ij < 4; ++ij) {
                k[t][b][ij >> 1][ij & 1] = (t == 0 ? sg[2 * b + (ij >> 1)] : 1.f) * em.em[t][(int64_t)ij * nblk + u.c[t][b]];
                acc[t * 8 + b * 4 + ij] = 0.0;
            }
    prior_kernel_done();
    const int64_t r0 = (int64_t)blockIdx.y * slice + sub, r1 = min(rows, (int64_t)(blockIdx.y + 1) * slice);
    unsigned char *ring_v = smem + sub * kRing * RowsV::kBytes, *ring_g = smem + kSubs * kRing * RowsV::kBytes + sub * kRing * RowsG::kBytes;
    const TV *pv = v + r0 * d;
    const TG *pg = g + r0 * d;
    float *w = g_out ? g_out + r0 * d + first : nullptr;
#pragma unroll 1
    for (int n = 0; n < kRing; ++n, pv += kSubs * d, pg += kSubs * d) {
        if (r0 + n * kSubs < r1) {
            RowsV::issue(ring_v + n * RowsV::kBytes, pv, u, s);
            RowsG::issue(ring_g + n * RowsG::kBytes, pg, u, s);
        }
        ring_commit();
    }
    int n = 0;
    for (int64_t r = r0; r < r1; r += kSubs, pv += kSubs * d, pg += kSubs * d, n = (n + 1) & (kRing - 1)) {
        float x[4], gy[4], y[4], z[4], h[4];
        double a[4], b[4];
        ring_wait();
        RowsV::first(ring_v + n * RowsV::kBytes, u, x);
        RowsG::second(ring_g + n * RowsG::kBytes, u, gy);
        __syncwarp();
        if (r + kRing * kSubs < r1) {
            RowsV::issue(ring_v + n * RowsV::kBytes, pv, u, s);
            RowsG::issue(ring_g + n * RowsG::kBytes, pg, u, s);
        }
        ring_commit();
        mul22<0, false>(x, k[0], y);           // x, y: states in front of the first and the second stage
        mul22<1, false>(y, k[1], z);
        u.transpose(words[sub][0], z);         // in front of the third
        if constexpr (NS == 4) {
            mul22<0, false>(z, k[2], h);       // in front of the fourth
            widen(h, a);
            widen(gy, b);
            outer22<1>(a, b, acc + 24);
            mul22<1, true>(gy, k[3], h);       // gradient behind the third
        } else {
#pragma unroll
            for (int i = 0; i < 4; ++i) h[i] = gy[i];
        }
        widen(z, a);
        widen(h, b);
        outer22<0>(a, b, acc + 16);
        mul22<0, true>(h, k[2], gy);
        u.transpose(words[sub][1], gy);        // behind the second
        widen(y, a);
        widen(gy, b);
        outer22<1>(a, b, acc + 8);
        mul22<1, true>(gy, k[1], h);           // behind the first
        widen(x, a);
        widen(h, b);
        outer22<0>(a, b, acc);
        if (w) {
            mul22<0, true>(h, k[0], gy);
            if (u.have) store_block<4>(w, s, S1, gy);
            w += kSubs * d;
        }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
#pragma unroll
    for (int e = 0; e < 8; ++e) acc[e] = sg[e >> 1] < 0.f ? -acc[e] : acc[e];        // [block][i][j]: coordinate 2 block + i
    combine<8 * NS, kSubs>(acc, reinterpret_cast<double (*)[kSubs][32]>(smem), sub, lane, add, [&](int e) -> double * {
        return !u.have ? nullptr : part.part[e >> 3] + ((int64_t)blockIdx.y * 4 + (e & 3)) * nblk + u.c[e >> 3][(e >> 2) & 1];
    });
}

// ---- two radix-2 stages of strides s and 2 s: a thread holds the four coordinates base + (i1 + 2 i2) s
struct Pair22 {
    int64_t base, c1[2], c2[2];        // block numbers: first stage at i2 = 0, 1, second stage at i1 = 0, 1
    bool have;
    __device__ __forceinline__ Pair22(int64_t d, int64_t s, int64_t unit) {
        have = unit < d / 4;
        const int64_t u = have ? unit : 0;
        const int64_t alpha = u / s, beta = u - alpha * s;
        base = alpha * 4 * s + beta;
        c1[0] = 2 * alpha * s + beta;
        c1[1] = c1[0] + s;
        c2[0] = 2 * alpha * s + beta;
        c2[1] = c2[0] + s;
    }
};

template <typename TI>
__global__ void __launch_bounds__(kOwnThreads)
fwd22_kernel(const TI *__restrict__ in, const int8_t *__restrict__ signs, int vec, float *__restrict__ out, int64_t rows, int64_t d, int64_t s,
             const float *__restrict__ em1, const float *__restrict__ em2) {
    const Pair22 u(d, s, (int64_t)blockIdx.x * kOwnThreads + threadIdx.x);
    if (!u.have) return;
    const int64_t nblk = d / 2;
    float k1[2][2][2], k2[2][2][2];
#pragma unroll
    for (int b = 0; b < 2; ++b)
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const float sg = sign_of(signs, u.base + (i + 2 * b) * s);
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                k1[b][i][j] = sg * em1[(int64_t)(i * 2 + j) * nblk + u.c1[b]];
                k2[b][i][j] = em2[(int64_t)(i * 2 + j) * nblk + u.c2[b]];
            }
        }
    prior_kernel_done();
    const int64_t r0 = (int64_t)blockIdx.y * kFwdRows, r1 = min(rows, r0 + kFwdRows);
    const TI *p = in + r0 * d + u.base;
    float *w = out + r0 * d + u.base;
    for (int64_t r = r0; r < r1; r += 4, p += 4 * d, w += 4 * d) {
        float x[4][4];
#pragma unroll
        for (int n = 0; n < 4; ++n)
            if (r + n < r1) load_block<4, TI>(p + n * d, s, vec, x[n]);
#pragma unroll
        for (int n = 0; n < 4; ++n) {
            if (r + n >= r1) break;
            float y[4], z[4];
#pragma unroll
            for (int b = 0; b < 2; ++b)
#pragma unroll
                for (int j = 0; j < 2; ++j) y[j + 2 * b] = fmaf(x[n][1 + 2 * b], k1[b][1][j], fmaf(x[n][2 * b], k1[b][0][j], 0.f));
#pragma unroll
            for (int b = 0; b < 2; ++b)
#pragma unroll
                for (int j = 0; j < 2; ++j) z[b + 2 * j] = fmaf(y[b + 2], k2[b][1][j], fmaf(y[b], k2[b][0][j], 0.f));
            store_block<4>(w + n * d, s, s == 1, z);
        }
    }
}

template <typename TV, typename TG>
__global__ void __launch_bounds__(32 * kSubs, 4)
bwd22_kernel(const TV *__restrict__ v, const int8_t *__restrict__ signs, int vec_v, const TG *__restrict__ g, int vec_g, float *__restrict__ g_out,
             int64_t rows, int64_t d, int64_t s, int slice, int add, const float *__restrict__ em1, const float *__restrict__ em2, double *__restrict__ part1,
             double *__restrict__ part2) {
    __shared__ double sh[16][kSubs][32];
    const int lane = threadIdx.x & 31, sub = threadIdx.x >> 5;
    const Pair22 u(d, s, (int64_t)blockIdx.x * 32 + lane);
    const int64_t nblk = d / 2;
    float k1[2][2][2], k2[2][2][2], sg[4];
    double acc[16];                            // first stage's sums [i2][i][j], second stage's [i1][i][j]
#pragma unroll
    for (int b = 0; b < 2; ++b)
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            sg[i + 2 * b] = sign_of(signs, u.base + (i + 2 * b) * s);
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                k1[b][i][j] = em1[(int64_t)(i * 2 + j) * nblk + u.c1[b]];
                k2[b][i][j] = em2[(int64_t)(i * 2 + j) * nblk + u.c2[b]];
                acc[b * 4 + i * 2 + j] = acc[8 + b * 4 + i * 2 + j] = 0.0;
            }
        }
    prior_kernel_done();
    const int64_t r0 = (int64_t)blockIdx.y * slice + sub, r1 = min(rows, (int64_t)(blockIdx.y + 1) * slice);
    constexpr int U = 2;
    for (int64_t r = r0; r < r1; r += U * kSubs) {
        float xx[U][4], gg[U][4];
#pragma unroll
        for (int n = 0; n < U; ++n)
            if (r + n * kSubs < r1) {
                load_block<4, TV>(v + (r + n * kSubs) * d + u.base, s, vec_v, xx[n]);
                load_block<4, TG>(g + (r + n * kSubs) * d + u.base, s, vec_g, gg[n]);
            }
#pragma unroll
        for (int n = 0; n < U; ++n) {
            if (r + n * kSubs >= r1) break;
            float x[4], y[4], h[4], o[4];
            double xd[4], yd[4], gd[4], hd[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) x[i] = sg[i] * xx[n][i];
#pragma unroll
            for (int b = 0; b < 2; ++b)
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    y[j + 2 * b] = fmaf(x[1 + 2 * b], k1[b][1][j], fmaf(x[2 * b], k1[b][0][j], 0.f));
                    // gradient behind the first stage: sum over the second stage's results
                    h[b + 2 * j] = fmaf(gg[n][b + 2], k2[b][j][1], fmaf(gg[n][b], k2[b][j][0], 0.f));
                }
#pragma unroll
            for (int i = 0; i < 4; ++i) { xd[i] = (double)x[i]; yd[i] = (double)y[i]; gd[i] = (double)gg[n][i]; hd[i] = (double)h[i]; }
#pragma unroll
            for (int b = 0; b < 2; ++b)
#pragma unroll
                for (int i = 0; i < 2; ++i)
#pragma unroll
                    for (int j = 0; j < 2; ++j) {
                        acc[8 + b * 4 + i * 2 + j] += yd[b + 2 * i] * gd[b + 2 * j];
                        acc[b * 4 + i * 2 + j] += xd[i + 2 * b] * hd[j + 2 * b];
                    }
            if (g_out && u.have) {
#pragma unroll
                for (int b = 0; b < 2; ++b)
#pragma unroll
                    for (int i = 0; i < 2; ++i) o[i + 2 * b] = fmaf(h[1 + 2 * b], k1[b][i][1], fmaf(h[2 * b], k1[b][i][0], 0.f));
                store_block<4>(g_out + (r + n * kSubs) * d + u.base, s, s == 1, o);
            }
        }
    }
    double *d1 = part1 + (int64_t)blockIdx.y * 4 * nblk, *d2 = part2 + (int64_t)blockIdx.y * 4 * nblk;
    combine<16, kSubs>(acc, sh, sub, lane, add, [&](int e) -> double * {
        if (!u.have) return nullptr;
        const int b = (e >> 2) & 1, ij = e & 3;
        return e < 8 ? d1 + (int64_t)ij * nblk + u.c1[b] : d2 + (int64_t)ij * nblk + u.c2[b];
    });
}

// ---- one radix-2 stage at a stride that is a multiple of four, backward: a thread owns four neighbouring blocks, so that a row is two 16-byte loads
// of either state where single blocks take 4-byte ones (1024 rows of d = 8192 behind four radix-8 stages: 30 us at 2.2 TB/s)
template <typename TV, typename TG>
__global__ void __launch_bounds__(32 * kSubs, 4)
bwd2x4_kernel(const TV *__restrict__ v, const TG *__restrict__ g, float *__restrict__ g_out, int64_t rows, int64_t d, int64_t s, int slice, int add,
              const float *__restrict__ em, double *__restrict__ part) {
    __shared__ double sh[16][kSubs][32];
    const int lane = threadIdx.x & 31, sub = threadIdx.x >> 5;
    const int64_t nblk = d / 2, cc = ((int64_t)blockIdx.x * 32 + lane) * 4;
    const bool have = cc < nblk;
    const int64_t c = have ? cc : 0, alpha = c / s, base = alpha * 2 * s + (c - alpha * s);
    float k[2][2][4];
    double acc[16] = {};                       // [i][j][block]
#pragma unroll
    for (int ij = 0; ij < 4; ++ij) load_block<4, float>(em + ij * nblk + c, 1, true, k[ij >> 1][ij & 1]);
    prior_kernel_done();
    const int64_t r0 = (int64_t)blockIdx.y * slice, r1 = min(rows, r0 + slice);
#pragma unroll 2
    for (int64_t r = r0 + sub; r < r1; r += kSubs) {
        float x[2][4], y[2][4];
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            load_block<4, TV>(v + r * d + base + i * s, 1, true, x[i]);
            load_block<4, TG>(g + r * d + base + i * s, 1, true, y[i]);
        }
        double xd[2][4], yd[2][4];
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int b = 0; b < 4; ++b) { xd[i][b] = (double)x[i][b]; yd[i][b] = (double)y[i][b]; }
#pragma unroll
        for (int ij = 0; ij < 4; ++ij)
#pragma unroll
            for (int b = 0; b < 4; ++b) acc[ij * 4 + b] += xd[ij >> 1][b] * yd[ij & 1][b];
        if (g_out && have) {
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                float o[4];
#pragma unroll
                for (int b = 0; b < 4; ++b) o[b] = fmaf(y[1][b], k[i][1][b], fmaf(y[0][b], k[i][0][b], 0.f));
                store_block<4>(g_out + r * d + base + i * s, 1, true, o);
            }
        }
    }
    double *dst = part + (int64_t)blockIdx.y * 4 * nblk + c;
    combine<16, kSubs>(acc, sh, sub, lane, add, [&](int e) -> double * { return have ? dst + (int64_t)(e >> 2) * nblk + (e & 3) : nullptr; });
}

// ---- one stage of radix 7, 8 or 16 on tiles in shared memory.  A CTA keeps NB neighbouring blocks and walks over tiles of eight rows that
// asynchronous copies bring into a ring of buffers; every value is fetched once, where threads that own entries of a block fetch all
// of the block's values.  Backward, the outer products of a block are a product of the fp64 tensor core (mma.m8n8k4, the rows as the
// contraction; radix 7 in an 8 x 8 tile): a lane converts one value of v and one of g where entry owners convert
// seventeen for two of theirs, and the sums take 2 registers an entry for 32 lanes together.
template <int B, bool S1, typename T>
struct Wide {
    static constexpr int NB = B <= 8 ? 32 : 16, NBW = NB / 4;          // blocks of a CTA, of a warp
    static constexpr int E = 16 / (int)sizeof(T);                      // elements of a copy
    static constexpr int kRows = 8;
    static constexpr int ST = S1 ? 1 : sizeof(T) == 4 ? NB + 4 : NB;   // from one value of a block to the next
    static constexpr int BP = !S1 ? 1 : sizeof(T) == 4 && B % 4 == 0 ? B + 4 : B;      // from one block to the next
    // rows apart: in fp32 eight banks (16-byte loads of four blocks for two values and four rows, 4-byte loads of eight values for four rows)
    static constexpr int pitch() {
        int rs = ((S1 ? NB * BP : B * ST) + E - 1) / E * E;
        if (sizeof(T) == 4) while (rs % 32 != 8) rs += 4;
        else rs += E;
        return rs;
    }
    static constexpr int RS = pitch(), kElems = kRows * RS;
    static constexpr int kPer = NB * B / E;                            // copies of a row; the CTA's threads are kGroup of them in kStep rows
    static constexpr int kGroup = kPer > 32 ? 64 : 32, kStep = kOwnThreads / kGroup;
    int64_t off;                       // of this thread's copies in a row, -1: none
    int to;
    __device__ __forceinline__ Wide(int64_t d, int64_t s) {
        const int k = (int)threadIdx.x % kGroup;
        const int64_t b0 = (int64_t)blockIdx.x * NB;
        off = -1;
        to = 0;
        if (k >= kPer) return;
        if constexpr (S1) {
            const int e = k * E;
            off = b0 * B + e;
            if (off >= d) off = -1;
            to = BP == B ? e : e / B * BP + e % B;
        } else {
            const int i = k / (NB / E), j = k % (NB / E) * E;
            const int64_t c = b0 + j, alpha = c / s;
            if (c < d / B) off = alpha * B * s + (c - alpha * s) + i * s;
            to = i * ST + j;
        }
    }
    // rows [r, r + 8) of the slice that ends at r1, zeros behind it
    __device__ __forceinline__ void issue(T *buf, const T *x, int64_t d, int64_t r, int64_t r1) const {
        if (off < 0) return;
        const int first = (int)threadIdx.x / kGroup;
#pragma unroll
        for (int n = 0; n < kRows; n += kStep) {
            const int64_t row = r + first + n;
            const uint32_t dst = (uint32_t)__cvta_generic_to_shared(buf + (first + n) * RS + to);
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(x + (row < r1 ? row : r1 - 1) * d + off), "r"(row < r1 ? 16 : 0) : "memory");
        }
    }
    // value i of four neighbouring blocks
    static __device__ __forceinline__ void four(const T *row, int i, int blk, float (&v)[4]) {
        if constexpr (S1) {
#pragma unroll
            for (int b = 0; b < 4; ++b) v[b] = to_f32<T>(row[(blk + b) * BP + i]);
        } else {
            load_block<4, T>(row + i * ST + blk, 1, true, v);
        }
    }
    // all values of a block
    static __device__ __forceinline__ void block(const T *row, int blk, float (&v)[B]) {
        load_block<B, T>(row + blk * BP, ST, S1 && (sizeof(T) == 2 || BP != B), v);
    }
};
// products of a block with IPL of its kernel's columns (forward) or rows (backward): lane -> block, results i0.. and rows first, first + step, ..
template <int B>
struct WideLane {
    static constexpr int IPL = 4;
    int blk, i0, first;
    static constexpr int step = 2;
    __device__ __forceinline__ WideLane() {
        const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
        if (B <= 8) { blk = 8 * w + (lane & 7); i0 = 4 * ((lane >> 3) & 1); first = lane >> 4; }
        else { blk = 8 * (w & 1) + (lane & 7); i0 = 4 * (lane >> 3); first = w >> 1; }
    }
};
template <int B, bool S1, typename T>
__device__ __forceinline__ void wide_products(const T *tile, const WideLane<B> &l, const float (&k)[4][B], float *out, int64_t d, int64_t s, int rows) {
#pragma unroll (B <= 8 ? 2 : 1)
    for (int n = 0; n < 4; ++n) {
        const int r = l.first + 2 * n;
        float v[B], o[4];
        Wide<B, S1, T>::block(tile + r * Wide<B, S1, T>::RS, l.blk, v);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            float a = 0.f;
#pragma unroll
            for (int j = 0; j < B; ++j) a = fmaf(v[j], k[i][j], a);
            o[i] = a;
        }
        if (out && r < rows) {
            float *p = out + (int64_t)r * d;
            if (S1 && B % 4 == 0) {
                *reinterpret_cast<float4 *>(p) = make_float4(o[0], o[1], o[2], o[3]);
            } else {
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    if (l.i0 + i < B) p[i * s] = o[i];
            }
        }
    }
}
constexpr int kWideFwdPerSm = 4, kWideBwdPerSm = 3, kWideStages = 3;

template <int B, bool S1, typename TI>
__global__ void __launch_bounds__(kOwnThreads, kWideFwdPerSm)
wide_fwd_kernel(const TI *__restrict__ in, const int8_t *__restrict__ signs, float *__restrict__ out, int64_t rows, int64_t d, int64_t s, int slice,
                const float *__restrict__ em) {
    using W = Wide<B, S1, TI>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    TI *buf = reinterpret_cast<TI *>(smem_raw);
    const W w(d, s);
    const WideLane<B> l;
    const int64_t nblk = d / B, c = (int64_t)blockIdx.x * W::NB + l.blk, cc = min(c, nblk - 1), alpha = cc / s, base = alpha * B * s + (cc - alpha * s);
    float k[4][B];
#pragma unroll
    for (int j = 0; j < B; ++j) {
        const float sg = sign_of(signs, base + j * s);
#pragma unroll
        for (int i = 0; i < 4; ++i) k[i][j] = l.i0 + i < B ? sg * em[(int64_t)(j * B + l.i0 + i) * nblk + cc] : 0.f;
    }
    prior_kernel_done();
    const int64_t r0 = (int64_t)blockIdx.y * slice, r1 = min(rows, r0 + slice);
    float *to = c < nblk ? out + base + l.i0 * s : nullptr;
    for (int n = 0; n < kWideStages - 1; ++n) {
        if (r0 + n * W::kRows < r1) w.issue(buf + n * W::kElems, in, d, r0 + n * W::kRows, r1);
        asm volatile("cp.async.commit_group;" ::: "memory");
    }
    int at = 0;
    for (int64_t r = r0; r < r1; r += W::kRows, at = at + 1 == kWideStages ? 0 : at + 1) {
        asm volatile("cp.async.wait_group %0;" ::"n"(kWideStages - 2) : "memory");
        __syncthreads();
        const int next = at == 0 ? kWideStages - 1 : at - 1;
        const int64_t rn = r + (kWideStages - 1) * W::kRows;
        if (rn < r1) w.issue(buf + next * W::kElems, in, d, rn, r1);
        asm volatile("cp.async.commit_group;" ::: "memory");
        wide_products<B, S1, TI>(buf + at * W::kElems, l, k, to ? to + r * d : nullptr, d, s, (int)min((int64_t)W::kRows, r1 - r));
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
}

__device__ __forceinline__ void dmma(double (&c)[2], double a, double b) {
    asm volatile("mma.sync.aligned.m8n8k4.row.col.f64.f64.f64.f64 {%0, %1}, {%2}, {%3}, {%0, %1};" : "+d"(c[0]), "+d"(c[1]) : "d"(a), "d"(b));
}

template <int B, bool S1, typename TV, typename TG>
__global__ void __launch_bounds__(kOwnThreads, kWideBwdPerSm)
wide_bwd_kernel(const TV *__restrict__ v, const int8_t *__restrict__ signs, const TG *__restrict__ g, float *__restrict__ g_out, int64_t rows, int64_t d,
                int64_t s, int slice, int add, const float *__restrict__ em, double *__restrict__ part) {
    using WV = Wide<B, S1, TV>;
    using WG = Wide<B, S1, TG>;
    constexpr int H = B <= 8 ? 1 : 2, Q = WV::NBW / 4, NB = WV::NB;    // 8 x 8 tiles of a block along either side; groups of four blocks of a warp
    extern __shared__ __align__(16) unsigned char smem_raw[];
    TV *buf_v = reinterpret_cast<TV *>(smem_raw);
    TG *buf_g = reinterpret_cast<TG *>(smem_raw + kWideStages * WV::kElems * sizeof(TV));
    const WV wv(d, s);
    const WG wg(d, s);
    const WideLane<B> l;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, kr = lane & 3, mi = lane >> 2;
    const int64_t nblk = d / B, c = (int64_t)blockIdx.x * NB + l.blk, cc = min(c, nblk - 1), alpha = cc / s, base = alpha * B * s + (cc - alpha * s);
    float k[4][B];
    if (!S1) {                             // (the gradient state in front of the first stage is not needed)
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < B; ++j) k[i][j] = l.i0 + i < B ? em[(int64_t)((l.i0 + i) * B + j) * nblk + cc] : 0.f;
    }
    double acc[Q][4][H][H][2] = {};
    prior_kernel_done();
    const int64_t r0 = (int64_t)blockIdx.y * slice, r1 = min(rows, r0 + slice);
    float *to = !S1 && g_out && c < nblk ? g_out + base + l.i0 * s : nullptr;
    for (int n = 0; n < kWideStages - 1; ++n) {
        if (r0 + n * 8 < r1) {
            wv.issue(buf_v + n * WV::kElems, v, d, r0 + n * 8, r1);
            wg.issue(buf_g + n * WG::kElems, g, d, r0 + n * 8, r1);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    }
    int at = 0;
    for (int64_t r = r0; r < r1; r += 8, at = at + 1 == kWideStages ? 0 : at + 1) {
        asm volatile("cp.async.wait_group %0;" ::"n"(kWideStages - 2) : "memory");
        __syncthreads();
        const int next = at == 0 ? kWideStages - 1 : at - 1;
        const int64_t rn = r + (kWideStages - 1) * 8;
        if (rn < r1) {
            wv.issue(buf_v + next * WV::kElems, v, d, rn, r1);
            wg.issue(buf_g + next * WG::kElems, g, d, rn, r1);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
        const TV *tv = buf_v + at * WV::kElems;
        const TG *tg = buf_g + at * WG::kElems;
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            const int b0 = warp * WV::NBW + 4 * q;
#pragma unroll
            for (int n = 0; n < 8; n += 4) {
                float a[H][4], b[H][4];
#pragma unroll
                for (int h = 0; h < H; ++h) {
                    const int i = min(8 * h + mi, B - 1);          // past the end of a radix of 7: entries that are not kept
                    WV::four(tv + (n + kr) * WV::RS, i, b0, a[h]);
                    WG::four(tg + (n + kr) * WG::RS, i, b0, b[h]);
                }
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    double bd[H];
#pragma unroll
                    for (int h = 0; h < H; ++h) bd[h] = (double)b[h][e];
#pragma unroll
                    for (int hi = 0; hi < H; ++hi) {
                        const double ad = (double)a[hi][e];
#pragma unroll
                        for (int hj = 0; hj < H; ++hj) dmma(acc[q][e][hi][hj], ad, bd[hj]);
                    }
                }
            }
        }
        if (!S1 && g_out) wide_products<B, S1, TG>(tg, l, k, to ? to + r * d : nullptr, d, s, (int)min((int64_t)8, r1 - r));
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    // by way of shared memory, [entry][block]: neighbouring threads add to neighbouring sums
    double *sums = reinterpret_cast<double *>(smem_raw);
#pragma unroll
    for (int q = 0; q < Q; ++q)
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int bl = warp * WV::NBW + 4 * q + e;
            const int64_t ce = min((int64_t)blockIdx.x * NB + bl, nblk - 1), al = ce / s, be = al * B * s + (ce - al * s);
#pragma unroll
            for (int hi = 0; hi < H; ++hi) {
                const int i = 8 * hi + mi;
                if (i >= B) continue;
                const bool neg = signs && signs[be + i * s] < 0;
#pragma unroll
                for (int hj = 0; hj < H; ++hj)
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const int j = 8 * hj + 2 * kr + h;
                        if (j < B) sums[(i * B + j) * (NB + 1) + bl] = neg ? -acc[q][e][hi][hj][h] : acc[q][e][hi][hj][h];
                    }
            }
        }
    __syncthreads();
    double *dst = part + (int64_t)blockIdx.y * (B * B) * nblk + (int64_t)blockIdx.x * NB;
    const int nb = (int)min((int64_t)NB, nblk - (int64_t)blockIdx.x * NB);
#pragma unroll 4
    for (int n = threadIdx.x; n < B * B * NB; n += kOwnThreads) {
        const int ij = n / NB, bl = n % NB;
        if (bl >= nb) continue;
        double *p = dst + (int64_t)ij * nblk + bl;
        const double x = sums[ij * (NB + 1) + bl];
        *p = add ? *p + x : x;
    }
}

// ---- sums over slices of all stages that keep partial sums: grad[c][i][j] (+)= sum over slices of part[slice][i b + j][c],
// slices in order, eight warps taking every eighth slice and their sums added in the order of the warps
struct ReduceStage { int64_t off, part_off, n_blk, total; int32_t bb, rows, n_slices; };
struct ReduceTable { int32_t m; int64_t total; ReduceStage st[HARP_MAX_STAGES]; };

__global__ void __launch_bounds__(kThreads)
reduce_kernel(const double *__restrict__ part, float *__restrict__ grad, int accumulate, const ReduceTable tab) {
    prior_kernel_done();
    __shared__ double warp_sum[kThreads / 32][32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    for (int64_t q0 = (int64_t)blockIdx.x * 32; q0 < tab.total; q0 += (int64_t)gridDim.x * 32) {
        int64_t q = q0 + lane;
        const bool have = q < tab.total;
        int t = 0;
        while (t + 1 < tab.m && q >= tab.st[t].total) { q -= tab.st[t].total; ++t; }
        const ReduceStage &s = tab.st[t];
        double sum = 0.0;
        if (have) {
            const double *p = part + s.part_off + q;
#pragma unroll 4
            for (int sl = w; sl < s.n_slices; sl += kThreads / 32) sum += p[(int64_t)sl * s.total];
        }
        warp_sum[w][lane] = sum;
        __syncthreads();
        if (w == 0 && have) {
            double all = warp_sum[0][lane];
            for (int k = 1; k < kThreads / 32; ++k) all += warp_sum[k][lane];
            const int64_t ij = q / s.n_blk, c = q - ij * s.n_blk;
            float *dst = grad + s.off + c * s.bb + ij;
            *dst = accumulate ? *dst + (float)all : (float)all;
        }
        __syncthreads();
    }
}

// ---- x with the permutation and the signs of the plan, rows of the same type: out[r][i] = s[perm[i]] x[r][perm[i]].  R rows at a
// time through shared memory (two elements of padding per 64 keep a digit reversal off the same banks), so that an index and
// its sign, twice the bytes of a bf16 row, are read once for all of them; staged = 0: rows too long for that are gathered from
// global memory one by one.  T: the bits of an element.  (2731 rows of d = 4096, bf16: 26 us with one row at a time, 17 with four)
template <typename T>
__global__ void __launch_bounds__(kThreads, 5)
permute_kernel(const T *__restrict__ x, int vec, T *__restrict__ out, int64_t rows, int d, const int32_t *__restrict__ perm,
               const int8_t *__restrict__ signs, int staged, int R) {
    prior_kernel_done();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T *tile = reinterpret_cast<T *>(smem_raw);
    constexpr int V = 16 / (int)sizeof(T);
    constexpr T kSignBit = (T)((T)1 << (8 * sizeof(T) - 1));
    const int pitch = (d + 2 * (d >> 6) + 2) / 2 * 2;
    for (int64_t r0 = (int64_t)blockIdx.x * R; r0 < rows; r0 += (int64_t)gridDim.x * R) {
        const int nr = (int)min((int64_t)R, rows - r0);
        const T *xr = x + r0 * d;
        T *outr = out + r0 * d;
        if (staged) {
            if (vec) {                                   // the rows are one run of 16-byte pieces
#pragma unroll 4
                for (int i = (int)threadIdx.x * V; i < nr * d; i += kThreads * V) {
                    const uint4 q = *reinterpret_cast<const uint4 *>(xr + i);
                    const int rr = (i >= d) + (i >= 2 * d) + (i >= 3 * d), c = i - rr * d;
                    uint32_t *dst = reinterpret_cast<uint32_t *>(tile + rr * pitch + c + 2 * (c >> 6));     // 4-byte aligned: the index is even
                    dst[0] = q.x; dst[1] = q.y; dst[2] = q.z; dst[3] = q.w;
                }
            } else {
                for (int rr = 0; rr < nr; ++rr)
                    for (int i = threadIdx.x; i < d; i += kThreads) tile[rr * pitch + i + 2 * (i >> 6)] = xr[(int64_t)rr * d + i];
            }
            __syncthreads();
        }
        auto gather = [&](const T *from, int step, bool padded) {
            if (d % 4 == 0) {
                for (int i = (int)threadIdx.x * 4; i < d; i += kThreads * 4) {
                    const int4 s4 = *reinterpret_cast<const int4 *>(perm + i);
                    int src[4] = {s4.x, s4.y, s4.z, s4.w};
                    T flip[4];
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        flip[k] = signs && signs[src[k]] < 0 ? kSignBit : (T)0;
                        if (padded) src[k] += 2 * (src[k] >> 6);
                    }
                    const T *f = from;
                    T *to = outr + i;
                    for (int rr = 0; rr < nr; ++rr, f += step, to += d) {
                        T o[4];
#pragma unroll
                        for (int k = 0; k < 4; ++k) o[k] = f[src[k]] ^ flip[k];
                        if constexpr (sizeof(T) == 2) *reinterpret_cast<uint2 *>(to) = make_uint2(o[0] | (uint32_t)o[1] << 16, o[2] | (uint32_t)o[3] << 16);
                        else *reinterpret_cast<uint4 *>(to) = make_uint4(o[0], o[1], o[2], o[3]);
                    }
                }
            } else {
                for (int i = threadIdx.x; i < d; i += kThreads) {
                    const int src = perm[i], at = padded ? src + 2 * (src >> 6) : src;
                    const T flip = signs && signs[src] < 0 ? kSignBit : (T)0;
                    for (int rr = 0; rr < nr; ++rr) outr[(int64_t)rr * d + i] = from[(int64_t)rr * step + at] ^ flip;
                }
            }
        };
        if (staged) gather(tile, pitch, true);
        else gather(xr, d, false);
        __syncthreads();
    }
}

// The same for aligned rows: groups of R rows by asynchronous 16-byte copies, the next group on its way while this one is gathered, and one table
// with the sign in its top bit in place of an index and the sign behind it.  harp_permute.h says where the pieces lie.
template <typename T>
__global__ void __launch_bounds__(kThreads, 3)
permute_ring_kernel(const T *__restrict__ x, T *__restrict__ out, int64_t rows, int d, const int32_t *__restrict__ table, int R) {
    constexpr int V = 16 / (int)sizeof(T);
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T *smem = reinterpret_cast<T *>(smem_raw);
    const int pieces = d / V, pitch = permute_pitch<V>(d);
    const int64_t groups = (rows + R - 1) / R;
    auto copy_in = [&](int64_t g, T *buf) {
        if (g < groups) {
            const int nr = (int)min((int64_t)R, rows - g * R);
            const T *src = x + g * R * d;
            for (int r = 0; r < nr; ++r)
#pragma unroll 2
                for (int c = threadIdx.x; c < pieces; c += kThreads)
                    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(buf + r * pitch + V * permute_piece<V>(c))), "l"(src + (int64_t)r * d + V * c) : "memory");
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    prior_kernel_done();
    copy_in(blockIdx.x, smem);
    int buf = 0;
    for (int64_t g = blockIdx.x; g < groups; g += gridDim.x, buf ^= 1) {
        copy_in(g + gridDim.x, smem + (buf ^ 1) * R * pitch);
        asm volatile("cp.async.wait_group 1;" ::: "memory");
        __syncthreads();
        const int nr = (int)min((int64_t)R, rows - g * R);
        const T *tile = smem + buf * R * pitch;
        for (int i = (int)threadIdx.x * 4; i < d; i += kThreads * 4) {
            const int4 t = __ldg(reinterpret_cast<const int4 *>(table + i));
            const int src[4] = {t.x, t.y, t.z, t.w};
            int at[4];
            T flip[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                at[k] = permute_place<V>(src[k] & 0x7fffffff);
                flip[k] = src[k] < 0 ? (T)((T)1 << (8 * sizeof(T) - 1)) : (T)0;
            }
            T *to = out + g * R * d + i;
            for (int r = 0; r < nr; ++r, to += d) {
                T o[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) o[k] = tile[r * pitch + at[k]] ^ flip[k];
                if constexpr (sizeof(T) == 2) *reinterpret_cast<uint2 *>(to) = make_uint2(o[0] | (uint32_t)o[1] << 16, o[2] | (uint32_t)o[3] << 16);
                else *reinterpret_cast<uint4 *>(to) = make_uint4(o[0], o[1], o[2], o[3]);
            }
        }
        __syncthreads();                                       // the buffer is free
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
}

// one stage on a chunk: out[r][base + j s] = sum_i in[r][base + i s] * K[c][i][j]   (transpose: K[c][j][i]).
// Neighbouring lanes hold neighbouring positions: inside one block when s is small, in neighbouring
// blocks otherwise -- so K is read block-major (entry k of block c at c b^2 + k) for s < 8 and
// element-major (at k D + c) from s = 8 on; kc_step / kk_step are the two strides of that choice.
template <typename TI>
__global__ void __launch_bounds__(kThreads)
stage_kernel(const TI *__restrict__ in, const int8_t *__restrict__ signs, float *__restrict__ out, int64_t rows, int64_t d, int b, int64_t s,
             const float *__restrict__ K, int64_t kc_step, int64_t kk_step, int transpose) {
    prior_kernel_done();
    // a thread keeps its position (the index arithmetic is done once) and walks over rows
    const int64_t pos = (int64_t)blockIdx.x * kThreads + threadIdx.x;
    if (pos >= d) return;
    const int64_t alpha = pos / (b * s), rem = pos - alpha * b * s;
    const int64_t j = rem / s, beta = rem - j * s;
    const int64_t base = alpha * b * s + beta;
    const float *Kc = K + (alpha * s + beta) * kc_step + (transpose ? j * b : j) * kk_step;
    const int64_t k_step = (transpose ? 1 : (int64_t)b) * kk_step;     // from K[..][i][j] to K[..][i+1][j] (or [j][i+1])
    for (int64_t r = blockIdx.y; r < rows; r += gridDim.y) {
        const TI *row = in + r * d + base;
        float acc = 0.f;
        for (int i = 0; i < b; ++i) {
            const float v = to_f32<TI>(row[(int64_t)i * s]);
            acc = fmaf(signs && signs[base + (int64_t)i * s] < 0 ? -v : v, Kc[(int64_t)i * k_step], acc);
        }
        out[r * d + pos] = acc;
    }
}

// grad[c][i][j] (+)= sum_r v[r][base_c + i s] * g[r][base_c + j s].  A CTA owns 32 neighbouring
// entries (one per lane); its eight warps take the rows r = w, w + 8, ... and their partial sums
// are added in a fixed order, so the result does not depend on scheduling.
// The 32 entries are neighbours within a block for s < 8 and the same entry of 32 neighbouring
// blocks from s = 8 on (by_block = 0), so that the lanes read neighbouring coordinates either way.
template <typename TV, typename TG>
__global__ void __launch_bounds__(kThreads)
outer_kernel(const TV *__restrict__ v, const int8_t *__restrict__ signs, const TG *__restrict__ g, int64_t rows, int64_t d, int b, int64_t s,
             float *__restrict__ grad, int accumulate, int by_block) {
    prior_kernel_done();
    __shared__ double part[kThreads / 32][32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int64_t total = d * b;                       // (d / b) blocks of b*b entries
    const int64_t nblk = d / b;
    for (int64_t e0 = (int64_t)blockIdx.x * 32; e0 < total; e0 += (int64_t)gridDim.x * 32) {
        const int64_t q = e0 + lane;
        int64_t e = q;
        double acc = 0.0;
        if (q < total) {
            const int64_t c = by_block ? q / (b * b) : q % nblk, ij = by_block ? q - c * b * b : q / nblk;
            e = c * b * b + ij;
            const int64_t i = ij / b, j = ij - i * b;
            const int64_t alpha = c / s, beta = c - alpha * s;
            const int64_t base = alpha * b * s + beta;
            const TV *pv = v + base + i * s;
            const TG *pg = g + base + j * s;
            for (int64_t r = w; r < rows; r += kThreads / 32) acc += (double)to_f32<TV>(pv[r * d]) * (double)to_f32<TG>(pg[r * d]);
            if (signs && signs[base + i * s] < 0) acc = -acc;
        }
        part[w][lane] = acc;
        __syncthreads();
        if (w == 0 && q < total) {
            double sum = part[0][lane];
            for (int k = 1; k < kThreads / 32; ++k) sum += part[k][lane];
            grad[e] = accumulate ? grad[e] + (float)sum : (float)sum;
        }
        __syncthreads();
    }
}

constexpr int64_t kMostScratch = 1280ll << 20, kLeastScratch = 160ll << 20;     // bytes of states of a chunk
// Bytes of one state of a chunk of a plan with one-thread-per-element kernels, which read two states once per row or column of a block: from L2, while
// they fit it (10000 rows of radices 7, 57, 4 6514 us in one chunk, 3577 in two; 1024 rows of 2^8, 49 1504 in one, of 51 MB, 1189 in two; 2048
// rows of 8, 8, 40, 2 behind a permutation 1466 in one, of 40 MB, and 1260 in two; 4096 rows of 2^8, 43 in bf16 3151 with 40 MB, 3229 with 32, 3861 with 16)
constexpr int64_t kPlainState = 32ll << 20;

// Scratch comes from a memory pool of the library's own (one per device, created on first use)
// that keeps one call's worth: the default pool hands its memory back at every
// synchronisation, and mapping 256 MB anew costs more than the kernels of a call.  What calls on several streams take beyond it goes back at a synchronisation.  Returns null
// if the pool cannot be created; the caller then allocates from the device's default pool.
cudaMemPool_t scratch_pool(int device) {
    static std::mutex mu;
    static std::map<int, cudaMemPool_t> pools;
    std::lock_guard<std::mutex> lock(mu);
    auto it = pools.find(device);
    if (it != pools.end()) return it->second;
    cudaMemPoolProps props = {};
    props.allocType = cudaMemAllocationTypePinned;
    props.handleTypes = cudaMemHandleTypeNone;
    props.location.type = cudaMemLocationTypeDevice;
    props.location.id = device;
    cudaMemPool_t pool = nullptr;
    if (cudaMemPoolCreate(&pool, &props) != cudaSuccess) {
        cudaGetLastError();
        pool = nullptr;
    } else {
        uint64_t keep = (uint64_t)kMostScratch + (256ull << 20);      // a call's states and partial sums
        cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &keep);
    }
    pools[device] = pool;
    return pool;
}

// grid of the kernels in which a thread keeps its coordinate and walks over rows
dim3 column_grid(int64_t d, int64_t rows) {
    const int64_t gx = (d + kThreads - 1) / kThreads;
    const int64_t gy = std::max<int64_t>(1, std::min<int64_t>(std::min<int64_t>(rows, 65535), (148 * 16 + gx - 1) / gx));
    return dim3((unsigned)gx, (unsigned)gy);
}

// ---- steps of a plan

struct Step { int t, n; bool wide; };  // stages [t, t + n): one stage, two of radix 4 or of radix 2, or three or four of radix 2; wide: one, on tiles in shared memory or by fours of blocks

// rows by asynchronous copies: eight neighbouring units are whole 16-byte pieces, the unit's sixteen coordinates make d a multiple of sixteen
bool aligned16(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }
bool ring44(int64_t s, const void *p) { return (s == 1 || s % 8 == 0) && aligned16(p); }

// Stages on tiles in shared memory: whole 16-byte pieces of neighbouring blocks, and rows enough for the tile of eight that they are worked on by
// (radices 16, 16, 16: 1 row 23.3 us on tiles, 21.1 without, 2 rows 23.4 and 24.0; 8, 8, 8, 8 in bf16: 3 rows 23.8 and 22.0, 6 rows 23.3 and 25.7).
bool wide_stage(const StageTable &st, int64_t d, int t, size_t es, const void *p, int64_t n_rows) {
    const int b = st.b[t];
    const int64_t e = 16 / (int64_t)es;
    return ((b == 16 && n_rows >= 2) || ((b == 7 || b == 8) && n_rows >= 4)) && (t == 0 ? d % e == 0 : st.s[t] % e == 0) && aligned16(p);
}

// a radix-2 stage alone, by fours of neighbouring blocks (the first stage, which carries the signs, has stride one) where they are a warp's worth: 8192
// rows of radices 2, 2, 2 25.1 us by fours, 21.8 by single blocks, of 4, 4, 2 27.7 and 24.6; 128 rows of 2, 2, 43, 2 36.6 and 40.7
bool fours_stage(const StageTable &st, int64_t d, int t, const void *p) { return st.b[t] == 2 && t > 0 && d >= 256 && st.s[t] % 4 == 0 && aligned16(p); }

// in, gy: the call's rows (the states of other steps start on 16-byte boundaries)
std::vector<Step> make_steps(const StageTable &st, int64_t d, size_t es, const void *in, const void *gy, int64_t n_rows) {
    std::vector<Step> steps;
    for (int t = 0; t < st.m;) {
        const int b = st.b[t];
        int n = 1;
        while (t + n < st.m && st.b[t + n] == b) ++n;
        // radix 2: threes in front so that fours are left over (d = 2048: 3 + 4 + 4; a three leaves a stride that is a multiple of eight behind it)
        const int k = n % 4 == 0 ? 4 : 3;
        const bool ring = b == 2 && n >= 3 && d % (16 * (int64_t)st.s[t]) == 0 && ring44(st.s[t], t == 0 ? in : nullptr) && aligned16(t + k == st.m ? gy : nullptr);
        n = ring ? k : n >= 2 && (b == 4 || b == 2) ? 2 : 1;
        const bool first = t == 0, last = t + n == st.m;
        const bool wide = wide_stage(st, d, t, first ? es : 4, first ? in : nullptr, n_rows) && wide_stage(st, d, t, last ? es : 4, last ? gy : nullptr, n_rows);
        steps.push_back({t, n, n == 1 && (wide || fours_stage(st, d, t, last ? gy : nullptr))});
        t += n;
    }
    return steps;
}

bool owner_radix(int b) { return (b >= 2 && b <= 8) || b == 16; }
// A backward kernel runs as one wave of CTAs, each with the largest number of rows that needs (a wave and a sixth takes as
// long as two: 2048 rows of d = 4096, 52 us with 128 rows per CTA): columns of CTAs, CTAs per SM -> rows per CTA
struct Shape { int64_t x; int per_sm; };
Shape bwd_shape(const harp_plan *plan, const Step &sp) {
    const int64_t d = plan->d;
    const int b = plan->st.b[sp.t];
    if (sp.wide && b == 2) return {(d / 2 + 127) / 128, 4};
    if (sp.wide) return {(d / b + (b <= 8 ? 31 : 15)) / (b <= 8 ? 32 : 16), kWideBwdPerSm};
    if (sp.n > 1) return b == 4 || sp.n > 2 ? Shape{(d / 16 + 7) / 8, k44PerSm} : Shape{(d / 4 + 31) / 32, 4};
    const int64_t x = (d / b + 31) / 32;
    switch (b) {
        case 7: return {x, bwd_per_sm(7, 4, 2)};
        case 8: return {x, bwd_per_sm(8, 2, 2)};
        case 16: return {x, bwd_per_sm(16, 2, 1)};
        case 5: return {x, bwd_per_sm(5, 5, kSubs)};
        case 6: return {x, bwd_per_sm(6, 3, kSubs)};
        default: return {x, bwd_per_sm(b, b, kSubs)};
    }
}
int slice_rows(const harp_plan *plan, const Step &sp, int64_t rows, int sms) {
    const Shape sh = bwd_shape(plan, sp);
    const int64_t y = std::max<int64_t>(1, sms * (int64_t)sh.per_sm / sh.x);
    // Narrow plans, whose wave has hundreds of slices: a slice's rows are a serial chain of the backward kernel, shared by `subs` warps, and
    // the slices one of the reduction, shared by eight; near the root of the rows the two last equally long (8192 rows of
    // d = 2: 592 slices 23.9 us, 158 slices 9.7)
    const int b = plan->st.b[sp.t], subs = sp.n > 1 || sp.wide ? kSubs : b == 16 ? 1 : b == 7 || b == 8 ? 2 : kSubs;
    const int64_t even = (int64_t)(0.125 * subs * std::sqrt((double)rows));
    const int64_t n = std::max<int64_t>(std::max<int64_t>(8, even), (rows + y - 1) / y);
    return (int)(sp.wide ? (n + 7) / 8 * 8 : n);
}
dim3 grid2(int64_t x, int per_x, int64_t rows, int per_y) { return dim3((unsigned)((x + per_x - 1) / per_x), (unsigned)((rows + per_y - 1) / per_y)); }

// The one-thread-per-element kernels read every state as often as a block has rows or columns, from L1 and L2.  An SM keeps the split of L1 and
// shared memory that the kernel before asked for, and behind the wide stages' 113 to 190 KB that is the smallest L1 (1024 rows of radices 7, 39, 2, 8:
// 1447 us, 718 this way; 128 rows 145 and 124); 14 percent, 32 KB, hold eight CTAs of 2 KB.  A small launch leaves the split alone (two rows of 4, 32, 4, 7:
// 53 us this way, 37).
Chain plain_chain(const Chain &chain, int64_t rows, int64_t d) { return {chain.stream, rows * d >= 1 << 17 ? 14 : -1}; }

// one step forward: out = in through the step's stages
template <typename TI>
void step_forward(const harp_plan *plan, const Step &sp, const TI *in, const int8_t *signs, float *out, int64_t rows, int sms, const Chain &st) {
    const int64_t d = plan->d, s = plan->st.s[sp.t];
    const int b = plan->st.b[sp.t];
    const float *em = plan->d_blocks_em + plan->st.off[sp.t];
    const float *em2 = sp.n == 2 ? plan->d_blocks_em + plan->st.off[sp.t + 1] : nullptr;
    const int vec = s == 1 && d % 4 == 0 && aligned16(in);
    if (sp.n > 2 || (sp.n == 2 && b == 4)) {
        // one wave of CTAs, like the backward kernels
        const int64_t x = (d / 16 + 8 * (kOwnThreads / 32) - 1) / (8 * (kOwnThreads / 32)), y = std::max<int64_t>(1, sms * (int64_t)kFwd44PerSm / x);
        const int slice = (int)std::max<int64_t>(kFwdRows / 2, (rows + y - 1) / y);
        const dim3 grid = grid2(d / 16, 8 * (kOwnThreads / 32), rows, slice);
        if (sp.n > 2) {
            Blocks4 k{};
            for (int t = 0; t < sp.n; ++t) k.em[t] = plan->d_blocks_em + plan->st.off[sp.t + t];
            auto go = [&](auto ns, auto s1) {
                launch_dep(fwd2222_kernel<decltype(ns)::value, decltype(s1)::value, TI>, grid, dim3(kOwnThreads), 0, st, in, signs, out, rows, d, s, slice, k);
            };
            using Three = std::integral_constant<int, 3>;
            using Four = std::integral_constant<int, 4>;
            if (sp.n == 4) s == 1 ? go(Four(), std::true_type()) : go(Four(), std::false_type());
            else s == 1 ? go(Three(), std::true_type()) : go(Three(), std::false_type());
            return;
        }
        auto go = [&](auto s1, auto ring) {
            launch_dep(fwd44_kernel<decltype(s1)::value, decltype(ring)::value, TI>, grid, dim3(kOwnThreads), 0, st, in, signs, vec, out, rows, d, s, slice, em, em2);
        };
        using std::true_type; using std::false_type;
        if (ring44(s, in)) s == 1 ? go(true_type(), true_type()) : go(false_type(), true_type());
        else s == 1 ? go(true_type(), false_type()) : go(false_type(), false_type());
        return;
    }
    if (sp.n == 2) {
        launch_dep(fwd22_kernel<TI>, grid2(d / 4, kOwnThreads, rows, kFwdRows), dim3(kOwnThreads), 0, st, in, signs, vec, out, rows, d, s, em, em2);
        return;
    }
    if (wide_stage(plan->st, d, sp.t, sizeof(TI), in, rows)) {
        auto go = [&](auto bc, auto s1) {
            constexpr int B = decltype(bc)::value;
            using W = Wide<B, decltype(s1)::value, TI>;
            const int64_t x = (d / B + W::NB - 1) / W::NB, y = std::max<int64_t>(1, sms * (int64_t)kWideFwdPerSm / x);
            const int slice = (int)((std::max<int64_t>(1, (rows + y - 1) / y) + 7) / 8 * 8);
            launch_dep(wide_fwd_kernel<B, decltype(s1)::value, TI>, dim3((unsigned)x, (unsigned)((rows + slice - 1) / slice)), dim3(kOwnThreads),
                       kWideStages * W::kElems * sizeof(TI), st, in, signs, out, rows, d, s, slice, em);
        };
        using std::true_type; using std::false_type;
        if (b == 7) s == 1 ? go(std::integral_constant<int, 7>(), true_type()) : go(std::integral_constant<int, 7>(), false_type());
        else if (b == 8) s == 1 ? go(std::integral_constant<int, 8>(), true_type()) : go(std::integral_constant<int, 8>(), false_type());
        else s == 1 ? go(std::integral_constant<int, 16>(), true_type()) : go(std::integral_constant<int, 16>(), false_type());
        return;
    }
#define HARP_FWD(B, OUT) case B: launch_dep(fwd_kernel<B, OUT, TI>, grid2(d / B, kOwnThreads / (B / OUT), rows, kFwdRows), dim3(kOwnThreads), 0, st, in, signs, vec, out, rows, d, s, em); return
    switch (b) {
        HARP_FWD(2, 2); HARP_FWD(3, 3); HARP_FWD(4, 4); HARP_FWD(5, 5); HARP_FWD(6, 6); HARP_FWD(7, 7); HARP_FWD(8, 4); HARP_FWD(16, 4);
        default: break;
    }
#undef HARP_FWD
    const bool by_em = s >= 8;                     // see stage_kernel
    launch_dep(stage_kernel<TI>, column_grid(d, rows), dim3(kThreads), 0, plain_chain(st, rows, d), in, signs, out, rows, d, b, s, by_em ? em : plan->d_blocks + plan->st.off[sp.t],
               by_em ? 1 : (int64_t)b * b, by_em ? d / b : 1, 0);
}

// one step backward: g_out (unless null) from g, sums of the step's outer products into part (or, radices without owner
// kernels, into grad)
template <typename TV, typename TG>
int step_backward(const harp_plan *plan, const Step &sp, const TV *v, const int8_t *signs, const TG *g, float *g_out, int64_t rows, double *all_parts, const int64_t *part_off,
                  int slice, int add, float *grad, int acc, const Chain &st) {
    const int64_t d = plan->d, s = plan->st.s[sp.t];
    const int b = plan->st.b[sp.t];
    const float *em = plan->d_blocks_em + plan->st.off[sp.t];
    const float *em2 = sp.n == 2 ? plan->d_blocks_em + plan->st.off[sp.t + 1] : nullptr;
    const int vec_v = s == 1 && d % 4 == 0 && aligned16(v), vec_g = s == 1 && d % 4 == 0 && aligned16(g);
    double *part = all_parts + part_off[sp.t], *part2 = sp.n == 2 ? all_parts + part_off[sp.t + 1] : nullptr;
    if (sp.n > 2) {
        const dim3 grid = grid2(d / 16, 8, rows, slice);
        Blocks4 k{};
        Sums4 sums{};
        for (int t = 0; t < sp.n; ++t) { k.em[t] = plan->d_blocks_em + plan->st.off[sp.t + t]; sums.part[t] = all_parts + part_off[sp.t + t]; }
        auto go = [&](auto ns, auto s1) {
            launch_dep(bwd2222_kernel<decltype(ns)::value, decltype(s1)::value, TV, TG>, grid, dim3(32 * kSubs), 0, st, v, signs, g, g_out, rows, d, s, slice, add, k, sums);
        };
        using Three = std::integral_constant<int, 3>;
        using Four = std::integral_constant<int, 4>;
        if (sp.n == 4) s == 1 ? go(Four(), std::true_type()) : go(Four(), std::false_type());
        else s == 1 ? go(Three(), std::true_type()) : go(Three(), std::false_type());
        return 1;
    }
    if (sp.n == 2 && b == 4) {
        const dim3 grid = grid2(d / 16, 8, rows, slice);
        auto go = [&](auto s1, auto ring) {
            launch_dep(bwd44_kernel<decltype(s1)::value, decltype(ring)::value, TV, TG>, grid, dim3(32 * kSubs), 0, st, v, signs, vec_v, g, vec_g, g_out, rows, d, s, slice, add, em, em2, part, part2);
        };
        using std::true_type; using std::false_type;
        if (ring44(s, v) && ring44(s, g)) s == 1 ? go(true_type(), true_type()) : go(false_type(), true_type());
        else s == 1 ? go(true_type(), false_type()) : go(false_type(), false_type());
        return 1;
    }
    if (sp.n == 2) {
        launch_dep(bwd22_kernel<TV, TG>, grid2(d / 4, 32, rows, slice), dim3(32 * kSubs), 0, st, v, signs, vec_v, g, vec_g, g_out, rows, d, s, slice, add, em, em2, part, part2);
        return 1;
    }
    if (sp.wide && b == 2) {
        launch_dep(bwd2x4_kernel<TV, TG>, grid2(d / 2, 128, rows, slice), dim3(32 * kSubs), 0, st, v, g, g_out, rows, d, s, slice, add, em, part);
        return 1;
    }
    if (sp.wide) {
        auto go = [&](auto bc, auto s1) {
            constexpr int B = decltype(bc)::value;
            using WV = Wide<B, decltype(s1)::value, TV>;
            using WG = Wide<B, decltype(s1)::value, TG>;
            const auto kern = wide_bwd_kernel<B, decltype(s1)::value, TV, TG>;
            const size_t smem = std::max(kWideStages * (WV::kElems * sizeof(TV) + WG::kElems * sizeof(TG)), sizeof(double) * B * B * (WV::NB + 1));      // the ring, then the sums
            // per call: the attribute belongs to the current device's copy of the kernel
            if (smem > 48 * 1024) cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
            launch_dep(kern, dim3((unsigned)((d / B + WV::NB - 1) / WV::NB), (unsigned)((rows + slice - 1) / slice)), dim3(kOwnThreads), smem, st,
                       v, signs, g, g_out, rows, d, s, slice, add, em, part);
        };
        using std::true_type; using std::false_type;
        if (b == 7) s == 1 ? go(std::integral_constant<int, 7>(), true_type()) : go(std::integral_constant<int, 7>(), false_type());
        else if (b == 8) s == 1 ? go(std::integral_constant<int, 8>(), true_type()) : go(std::integral_constant<int, 8>(), false_type());
        else s == 1 ? go(std::integral_constant<int, 16>(), true_type()) : go(std::integral_constant<int, 16>(), false_type());
        return 1;
    }
#define HARP_BWD(B, BI, SUBS) case B: launch_dep(bwd_kernel<B, BI, SUBS, TV, TG>, grid2(d / B, 32, rows, slice), dim3(32 * ((B + BI - 1) / BI) * SUBS), 0, st, v, signs, vec_v, g, vec_g, g_out, rows, d, s, slice, add, em, part); return 1
    switch (b) {
        HARP_BWD(2, 2, kSubs); HARP_BWD(3, 3, kSubs); HARP_BWD(4, 4, kSubs); HARP_BWD(5, 5, kSubs); HARP_BWD(6, 3, kSubs); HARP_BWD(7, 4, 2);
        HARP_BWD(8, 2, 2); HARP_BWD(16, 2, 1);
        default: break;
    }
#undef HARP_BWD
    const bool by_em = s >= 8;
    launch_dep(outer_kernel<TV, TG>, dim3((unsigned)std::min<int64_t>((d * b + 31) / 32, 148 * 64)), dim3(kThreads), 0, plain_chain(st, rows, d), v, signs, g, rows, d, b, s,
               grad + plan->st.off[sp.t], acc, by_em ? 0 : 1);
    if (!g_out) return 1;
    launch_dep(stage_kernel<TG>, column_grid(d, rows), dim3(kThreads), 0, plain_chain(st, rows, d), g, (const int8_t *)nullptr, g_out, rows, d, b, s,
               by_em ? em : plan->d_blocks + plan->st.off[sp.t], by_em ? 1 : (int64_t)b * b, by_em ? d / b : 1, 1);
    return 2;
}

template <typename T>
harp_status_t grad_blocks(const harp_plan *plan, const T *x, const T *gy, int64_t n_rows, float *grad, int accumulate, cudaStream_t stream) {
    const int64_t d = plan->d;
    const StageTable &tab = plan->st;
    const std::vector<Step> steps = make_steps(tab, d, sizeof(T), plan->d_perm ? nullptr : x, gy, n_rows);
    const int n = (int)steps.size(), n_g = std::min(n - 1, 2), ring = std::max(1, n_g);
    const bool permuted = plan->d_perm != nullptr;
    // Chunk of rows whose forward states, gradient states and permuted rows fit the budget; the partial sums of a wave of CTAs come on top.  The
    // forward kernels (none where one step is all) take kFwdRows rows per CTA along grid.y.  Chunks that stay near L2 are not worth their launches
    // and partial waves (16384 rows of d = 4096, call after call on the same rows: chunks of 110 MB 1083 us, 200 MB 863, 640 MB 751, one of 1200 MB 719; on others each time 777); a device without room for it takes the smaller ones.
    const int64_t per_row = std::max<int64_t>(1, d * (4 * (int64_t)(n - 1 + n_g) + (permuted ? (int64_t)sizeof(T) : 0)));
    int sms = 148;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, plan->device);
    int64_t chunk = 0, plane = 0, part_len = 0, part_off[HARP_MAX_STAGES] = {};
    ReduceTable red{};
    double *part = nullptr;
    cudaMemPool_t pool = scratch_pool(plan->device);
    const bool plain = std::any_of(steps.begin(), steps.end(), [&](const Step &sp) { return !owner_radix(tab.b[sp.t]); });
    for (int64_t budget = kMostScratch; !part; budget /= 2) {
        if (budget < kLeastScratch) return HARP_ERR_ALLOC;
        const int64_t fit = std::max<int64_t>(16, std::min(budget / per_row, plain ? kPlainState / (4 * d) : INT64_MAX)), most = n > 1 ? std::min<int64_t>(fit, 65535ll * kFwdRows) : fit;
        const int64_t n_chunks = (n_rows + most - 1) / most;
        chunk = (n_rows + n_chunks - 1) / n_chunks;
        part_len = 0;
        red = ReduceTable{};
        for (const Step &sp : steps) {
            const int b = tab.b[sp.t];
            if (!owner_radix(b)) continue;
            const int slice = slice_rows(plan, sp, chunk, sms);
            for (int t = sp.t; t < sp.t + sp.n; ++t) {
                part_off[t] = part_len;
                red.st[red.m++] = ReduceStage{tab.off[t], part_len, d / b, d * b, b * b, slice, 0};
                red.total += d * b;
                part_len += ((chunk + slice - 1) / slice) * d * b;
            }
        }
        plane = (chunk * d + 3) / 4 * 4;
        const int64_t states = plane * 4 * (n - 1 + n_g) + (permuted ? plane * (int64_t)sizeof(T) : 0);
        if (states > plan->opt_grad_scratch) continue;
        const size_t bytes = (size_t)(part_len * 8 + 16 + states);
        if ((pool ? cudaMallocFromPoolAsync(reinterpret_cast<void **>(&part), bytes, pool, stream) : cudaMallocAsync(reinterpret_cast<void **>(&part), bytes, stream)) != cudaSuccess) {
            cudaGetLastError();
            part = nullptr;
        }
    }
    float *vp = reinterpret_cast<float *>(part + (part_len + 1) / 2 * 2), *gp = vp + (n - 1) * plane;      // state planes on 16-byte boundaries
    T *xp = reinterpret_cast<T *>(gp + n_g * plane);
    const int8_t *signs = permuted ? nullptr : plan->d_signs;       // the permutation kernel carries the signs
    // a small call's kernels share one split (2400 rows of radices 4, 4, 4 behind a permutation 31.6 us each with its own, 22.3 this way; 256 rows of 2^11
    // 36.7 and 30.7); from some 2^22 values on it makes no difference or the larger L1 gains (16384 rows of d = 4096 708 and 716)
    const Chain st{stream, !plain && chunk * d <= 1 << 22 ? 100 : -1};
    harp_status_t rc = HARP_OK;
    for (int64_t r0 = 0; r0 < n_rows && rc == HARP_OK; r0 += chunk) {
        const int64_t rows = std::min(chunk, n_rows - r0);
        const int acc = accumulate || r0 > 0 ? 1 : 0;
        const T *xc = x + r0 * d, *gc = gy + r0 * d;
        int launches = 0;
        if (permuted) {
            using Bits = std::conditional_t<sizeof(T) == 2, uint16_t, uint32_t>;
            const size_t row_smem = (size_t)((d + 2 * (d >> 6) + 2) / 2 * 2) * sizeof(T);
            // four rows per CTA (the kernel counts on at most that) where they leave two CTAs for every SM (8 rows of d = 3375: the call 45.0 us
            // with four, 41.8 with one).  Shared memory is taken from the L1 that the one-thread-per-element kernels behind this one live on (radices 6, 54,
            // 20, 1024 rows: 3160 us behind 53 KB a CTA, 1750 behind 26; 7, 49, 8, 2051 rows in fp32: 2240 behind 44 KB, 1310 behind 11).
            const size_t cap = red.m == tab.m ? 100 * 1024 : 12 * 1024;
            int R = 4;
            while (R > 1 && (R * row_smem > cap || rows < 2 * (int64_t)R * sms)) R /= 2;
            size_t smem = R * row_smem;
            // per call: the attribute belongs to the current device's copy of the kernel
            const int staged = smem <= 48 * 1024 || (smem <= 200 * 1024 && cudaFuncSetAttribute(permute_kernel<Bits>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024) == cudaSuccess);
            if (!staged) smem = 0;
            const int32_t *table = harp_f32_source_table(plan);
            constexpr int V = 16 / (int)sizeof(T);
            const int64_t pitch_bytes = d % V == 0 ? permute_pitch<V>(d) * (int64_t)sizeof(T) : 0, ring_rows = pitch_bytes > 0 ? std::min<int64_t>(4, 36 * 1024 / pitch_bytes) : 0;
            if (table && red.m == tab.m && ring_rows > 0 && aligned16(xc)) {
                const int r = (int)std::max<int64_t>(1, std::min<int64_t>(ring_rows, rows / (3 * sms)));
                const size_t bytes = (size_t)(2 * r * pitch_bytes);
                if (bytes > 48 * 1024) cudaFuncSetAttribute(permute_ring_kernel<Bits>, cudaFuncAttributeMaxDynamicSharedMemorySize, 72 * 1024);
                launch_dep(permute_ring_kernel<Bits>, dim3((unsigned)std::min<int64_t>((rows + r - 1) / r, 3 * sms)), dim3(kThreads), bytes, st, reinterpret_cast<const Bits *>(xc),
                           reinterpret_cast<Bits *>(xp), rows, (int)d, table, r);
            } else {
                launch_dep(permute_kernel<Bits>, dim3((unsigned)std::min<int64_t>((rows + R - 1) / R, 148 * 8)), dim3(kThreads), smem, st, reinterpret_cast<const Bits *>(xc), (int)(aligned16(xc) && d % (16 / (int64_t)sizeof(T)) == 0), reinterpret_cast<Bits *>(xp),
                       rows, (int)d, plan->d_perm, plan->d_signs, staged, R);
            }
            xc = xp;
            ++launches;
        }
        for (int k = 0; k + 1 < n; ++k, ++launches) {
            if (k == 0) step_forward<T>(plan, steps[0], xc, signs, vp, rows, sms, st);
            else step_forward<float>(plan, steps[(size_t)k], vp + (k - 1) * plane, nullptr, vp + k * plane, rows, sms, st);
        }
        for (int k = n - 1; k >= 0; --k) {
            const Step &sp = steps[(size_t)k];
            const float *v_in = vp + (k - 1) * plane, *g_in = gp + ((k + 1) % ring) * plane;
            float *out = k > 0 ? gp + (k % ring) * plane : nullptr;
            const int slice = slice_rows(plan, sp, chunk, sms);
            if (k == 0 && k == n - 1) launches += step_backward<T, T>(plan, sp, xc, signs, gc, out, rows, part, part_off, slice, r0 > 0, grad, acc, st);
            else if (k == n - 1) launches += step_backward<float, T>(plan, sp, v_in, nullptr, gc, out, rows, part, part_off, slice, r0 > 0, grad, acc, st);
            else if (k == 0) launches += step_backward<T, float>(plan, sp, xc, signs, g_in, out, rows, part, part_off, slice, r0 > 0, grad, acc, st);
            else launches += step_backward<float, float>(plan, sp, v_in, nullptr, g_in, out, rows, part, part_off, slice, r0 > 0, grad, acc, st);
        }
        if (red.m > 0 && r0 + chunk >= n_rows) {
            for (int k = 0; k < red.m; ++k) red.st[k].n_slices = (int32_t)((chunk + red.st[k].rows - 1) / red.st[k].rows);
            launch_dep(reduce_kernel, dim3((unsigned)std::min<int64_t>((red.total + 31) / 32, 148 * 16)), dim3(kThreads), 0, st, part, grad, accumulate, red);
            ++launches;
        }
        g_harp_launches.fetch_add(launches, std::memory_order_relaxed);
        if (cudaGetLastError() != cudaSuccess) rc = HARP_ERR_CUDA;
    }
    cudaFreeAsync(part, stream);
    return rc;
}

}  // namespace

extern "C" int64_t harp_plan_n_params(const harp_plan_t *plan) { return plan ? plan->n_params : -1; }

extern "C" harp_status_t harp_grad_blocks(const harp_plan_t *plan, const void *x, const void *gy, int64_t n_rows,
                                          harp_dtype_t dtype, float *grad, int accumulate, void *stream) {
    if (!plan || !grad) return HARP_ERR_NULL;
    if (dtype != HARP_F32 && dtype != HARP_BF16) return HARP_ERR_BAD_DTYPE;
    {
        int dev = -1;
        if (cudaGetDevice(&dev) != cudaSuccess) return HARP_ERR_CUDA;
        if (dev != plan->device) return HARP_ERR_DIM_MISMATCH;      // the scratch pool and the plan's tables live on plan->device
    }
    if (n_rows < 0) return HARP_ERR_BAD_DIM;
    if (n_rows > 0 && (!x || !gy)) return HARP_ERR_NULL;
    const size_t es = harp_dtype_size(dtype);
    if (reinterpret_cast<uintptr_t>(x) % es || reinterpret_cast<uintptr_t>(gy) % es || reinterpret_cast<uintptr_t>(grad) % 4)
        return HARP_ERR_BAD_DIM;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (n_rows == 0) {
        if (!accumulate && cudaMemsetAsync(grad, 0, sizeof(float) * (size_t)plan->n_params, st) != cudaSuccess) return HARP_ERR_CUDA;
        return HARP_OK;
    }
    return dtype == HARP_F32 ? grad_blocks<float>(plan, (const float *)x, (const float *)gy, n_rows, grad, accumulate, st)
                             : grad_blocks<__nv_bfloat16>(plan, (const __nv_bfloat16 *)x, (const __nv_bfloat16 *)gy, n_rows, grad, accumulate, st);
}
