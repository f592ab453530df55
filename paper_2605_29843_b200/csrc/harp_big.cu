// fp32 rows, one strided stage of radix 17 to 48: a register-tiled product per block.
//
// A tile is R rows x b places x 8 neighbouring positions (32-byte runs of the rows), brought and taken by bulk tensor copies, 32-byte
// swizzle, three buffers; the block kernels of the eight positions stay in shared memory while a CTA keeps its positions.  A warp multiplies
// four neighbouring blocks (lane / 8) by JT of their results each: a lane holds RT rows (lane % 8 + 8 k) x JT results, so that a value is fetched
// once per JT products and a kernel entry once per RT, where lanes that share one kernel and hold two rows each (the passes of harp_f32.cu) spend
// a broadcast fetch of four entries on eight products and are bound by it: 4096 rows of d = 11008, radix 43: 278 us.  The 32 lanes' values
// are on different banks, for the operands as for the results.
//
// What bounds it: the products (43 of 48 results kept) and the copy engine (a run of 32 bytes in and out takes 3.3 cycles), about equally.
// All positions of some rows are worked on at the same time, a CTA to eight of them, for the sake of DRAM pages (an equal share of the whole list of
// tiles for each of 148 SMs instead of 128: 287 us for both passes of 4096 rows of d = 11008, 186 this way).
#include <algorithm>

#include "harp_internal.h"
#include "harp_regs.h"
#include "harp_ring.h"
#include "harp_tm_ptx.cuh"

namespace {

using harp_tm::smem_u32;

constexpr int kBigWarps = 8, kBigThreads = 32 * (kBigWarps + 1);       // the last warp copies
constexpr uint32_t kBigSpin = 1u << 22;        // limit of every wait for a bulk copy
constexpr int kBigSmem = 226 * 1024, kBigBufs = 3;

struct BigArgs {
    int32_t b, pitch;          // radix; floats per row of a kernel in shared memory
    int32_t n_lo, n_cg;        // groups of eight positions below the stride, of the plan
    int32_t n_tiles, n_parts;  // tiles along the rows; a CTA takes every n_parts-th of its group
    int64_t S, off;            // stride of the stage, its offset in the block array
};

template <int JT, int RT, bool TR>
__global__ void __launch_bounds__(kBigThreads, 1)
harp_big_kernel(const float *__restrict__ blocks, int32_t *err, const __grid_constant__ CUtensorMap tmap, const BigArgs P) {
    constexpr int R = 8 * RT;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ __align__(8) uint64_t full_bar[kBigBufs], done_bar[kBigBufs];       // the tile has arrived; the warps have stored its results
    __shared__ int dead;
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");        // (whoever comes next waits for this grid's end before it touches a row)
    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u, tile_bytes = (uint32_t)P.b * R * 32u;
    float *wts = reinterpret_cast<float *>(smem_raw + (base - smem_u32(smem_raw)) + kBigBufs * tile_bytes);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, rl = lane & 7, l = 4 * (warp >> 2) + (lane >> 3), j0 = (warp & 3) * JT;
    const int b = P.b, pitch = P.pitch;
    if (threadIdx.x == 0) {
        for (int k = 0; k < kBigBufs; ++k) { harp_tm::mbar_init(smem_u32(&full_bar[k]), 1); harp_tm::mbar_init(smem_u32(&done_bar[k]), kBigWarps); }
        dead = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    const int g = blockIdx.x % P.n_cg, t0 = blockIdx.x / P.n_cg, hi = g / P.n_lo, lo = g - hi * P.n_lo;
    const int n_my = t0 < P.n_tiles ? (P.n_tiles - t0 + P.n_parts - 1) / P.n_parts : 0;
    __syncthreads();
    if (n_my > 0) {                                            // the kernels of the eight positions, [position][operand][result]
        const float *src = blocks + P.off + ((int64_t)hi * P.S + lo * 8) * b * b;      // neighbouring blocks are neighbours in memory
        for (int k = 0; k < 8; ++k)                            // a warp per row of a kernel
            for (int i = warp; i < b; i += kBigThreads / 32)
                for (int j = lane; j < b; j += 32)
                    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_u32(wts + (k * b + (TR ? j : i)) * pitch + (TR ? i : j))), "l"(src + (k * b + i) * b + j) : "memory");
    }
    auto stopped = [&] { return *(volatile int *)&dead != 0; };
    // whether the phase of a barrier completed before the limit; after one that did not nothing is copied any more
    auto wait = [&](uint64_t *bar, uint32_t parity) {
        for (uint32_t it = 0; !harp_tm::mbar_try(smem_u32(bar), parity);)
            if (++it > kBigSpin || ((it & 63) == 63 && stopped())) {
                *(volatile int *)&dead = 1;
                atomicExch(err, 103);
                return;
            }
    };
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    // plan data only up to here: may run under the kernel before this one
    asm volatile("griddepcontrol.wait;" ::: "memory");

    if (warp == kBigWarps) {                                   // copies; tile n in buffer n mod kBigBufs
        if (lane != 0) return;
        uint32_t loaded = ~0u;                                 // bit per buffer: phase of its last load
        auto load = [&](int n) {
            const int k = n % kBigBufs;
            harp_tm::mbar_expect_tx(smem_u32(&full_bar[k]), tile_bytes);       // past the last row the engine fills zeros
            harp_tm::tma_load_3d(base + k * tile_bytes, &tmap, lo * 8, (t0 + n * P.n_parts) * R, hi * b, smem_u32(&full_bar[k]));
            loaded ^= 1u << k;
        };
        for (int n = 0; n < kBigBufs && n < n_my; ++n) load(n);
        for (int n = 0; n < n_my && !stopped(); ++n) {
            const int k = n % kBigBufs;
            wait(&done_bar[k], (uint32_t)(n / kBigBufs) & 1u);
            if (stopped()) break;
            harp_tm::tma_store_3d(&tmap, lo * 8, (t0 + n * P.n_parts) * R, hi * b, base + k * tile_bytes);
            harp_tm::bulk_commit();
            if (n + kBigBufs < n_my) {
                harp_tm::bulk_wait_read0();
                load(n + kBigBufs);
            }
        }
        harp_tm::bulk_wait0();
        if (stopped()) ring_drain(loaded, kBigBufs, kBigSpin, [&](int k, uint32_t phase) { return harp_tm::mbar_try(smem_u32(&full_bar[k]), phase); });
        return;
    }

    // byte offset of (position l, row lane % 8) in a place of the tile: 16-byte halves exchanged in every second group of four rows
    const uint32_t at0 = (uint32_t)(rl * 32 + ((l * 4) ^ (((rl >> 2) & 1) << 4)));
    for (int n = 0; n < n_my; ++n) {
        const int buf = n % kBigBufs;
        wait(&full_bar[buf], (uint32_t)(n / kBigBufs) & 1u);
        const uint32_t tile = base + buf * tile_bytes + at0;
        const float *w = wts + (size_t)l * b * pitch + j0;
        float acc[JT][RT] = {};
        // values and kernel entries of an operand; those of the next one are fetched under its products
        struct Operand { float x[RT]; float4 k[JT / 4]; } oa, ob;
        auto fetch = [&](Operand &o, int i) {
#pragma unroll
            for (int k = 0; k < RT; ++k) asm volatile("ld.shared.f32 %0, [%1];" : "=f"(o.x[k]) : "r"(tile + (uint32_t)i * (R * 32) + k * 256) : "memory");
#pragma unroll
            for (int j = 0; j < JT / 4; ++j) o.k[j] = *reinterpret_cast<const float4 *>(w + i * pitch + 4 * j);
        };
        auto multiply = [&](const Operand &o) {
#pragma unroll
            for (int j = 0; j < JT; ++j) {
                const float4 &q = o.k[j / 4];
                const float e = j % 4 == 0 ? q.x : j % 4 == 1 ? q.y : j % 4 == 2 ? q.z : q.w;
#pragma unroll
                for (int k = 0; k < RT; ++k) acc[j][k] = fmaf(o.x[k], e, acc[j][k]);
            }
        };
        fetch(oa, 0);
        for (int i = 0; i + 1 < b; i += 2) {
            fetch(ob, i + 1);
            multiply(oa);
            fetch(oa, min(i + 2, b - 1));
            multiply(ob);
        }
        if (b & 1) multiply(oa);
        // nobody stores before everybody has read: the four warps that share these positions
        asm volatile("bar.sync %0, 128;" ::"r"(1 + (warp >> 2)) : "memory");
#pragma unroll
        for (int j = 0; j < JT; ++j)
            if (j0 + j < b) {
#pragma unroll
                for (int k = 0; k < RT; ++k)
                    asm volatile("st.shared.f32 [%0], %1;" ::"r"(tile + (uint32_t)(j0 + j) * (R * 32) + k * 256), "f"(acc[j][k]) : "memory");
            }
        harp_tm::fence_async_smem();                           // results before the copy engine reads them
        __syncwarp();
        if (lane == 0) harp_tm::mbar_arrive(smem_u32(&done_bar[buf]));
    }
}

typedef CUresult (*EncodeTiled)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *, const cuuint64_t *,
                                const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle,
                                CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

int big_pitch(int b) { return (b + 3) / 4 * 4; }
int64_t big_smem(int b, int rt) {              // the tiles, the kernels and what a lane reads past the last of them
    return 1024 + kBigBufs * (int64_t)b * rt * 256 + 8 * (int64_t)b * big_pitch(b) * 4 + 64;
}

template <int JT, int RT, bool TR>
cudaError_t launch(void *encode, const RegPass &P, int b, int sms, float *x, int64_t n, int64_t ld, const float *blocks, int32_t *err, cudaStream_t stream) {
    constexpr int R = 8 * RT;
    CUtensorMap tmap = {};
    // (position below the stride, row, place)
    const cuuint64_t gdim[3] = {(cuuint64_t)P.S, (cuuint64_t)n, (cuuint64_t)(P.d / P.S)}, gstr[2] = {(cuuint64_t)ld * 4, (cuuint64_t)P.S * 4};
    const cuuint32_t box[3] = {8, R, (cuuint32_t)b}, ones[3] = {1, 1, 1};
    if (reinterpret_cast<EncodeTiled>(encode)(&tmap, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, x, gdim, gstr, box, ones, CU_TENSOR_MAP_INTERLEAVE_NONE,
                                              CU_TENSOR_MAP_SWIZZLE_32B, CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
        return cudaErrorInvalidValue;
    const auto kern = harp_big_kernel<JT, RT, TR>;
    const int64_t smem = big_smem(b, RT);
    const cudaError_t ae = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kBigSmem);
    if (ae != cudaSuccess) return ae;
    BigArgs A{b, big_pitch(b), P.n_lo, P.n_cg, (int32_t)((n + R - 1) / R), 0, P.S, P.off[0]};
    A.n_parts = (int32_t)std::max<int64_t>(1, std::min<int64_t>(A.n_tiles, sms / A.n_cg));
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(A.n_parts * A.n_cg));
    cfg.blockDim = dim3(kBigThreads);
    cfg.dynamicSmemBytes = (size_t)smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, blocks, err, tmap, A);
}

}  // namespace

// Stage t of the plan as a pass over rows, if there is a kernel for it.
bool harp_big_pass(const StageTable &st, int64_t d, int t, RegPass &P) {
    const int b = st.b[t];
    const int64_t S = st.s[t];
    // up to 48 results for the twelve of a lane and four warps
    if (b <= 16 || b > 48 || S % 8 != 0) return false;
    P = RegPass{};
    P.shape = kBigShape + b;
    P.S = S;
    P.d = d;
    P.n_lo = (int32_t)(S / 8);
    P.n_cg = (int32_t)(d / b / 8);
    P.off[0] = st.off[t];
    return true;
}

cudaError_t harp_big_launch(void *encode, const RegPass &P, int sms, float *x, int64_t n, int64_t ld, const float *blocks, int transpose, int32_t *err, cudaStream_t stream) {
    const int b = P.shape - kBigShape;
#define HARP_BIG(JT, RT) (transpose ? launch<JT, RT, true>(encode, P, b, sms, x, n, ld, blocks, err, stream) : launch<JT, RT, false>(encode, P, b, sms, x, n, ld, blocks, err, stream))
    // as many rows as three buffers beside the kernels leave room for
    if (b <= 32) return HARP_BIG(8, 8);
    if (big_smem(b, 6) <= kBigSmem) return HARP_BIG(12, 6);
    if (big_smem(b, 5) <= kBigSmem) return HARP_BIG(12, 5);
    return HARP_BIG(12, 4);
#undef HARP_BIG
}
