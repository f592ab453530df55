// Host-side helpers shared by the tensor-core plan builders: stage grouping, fused block
// matrices (fp64), bf16 rounding, and the slot maps of the mma.sync operand layouts.
#pragma once

#include <cstring>
#include <vector>

#include "harp_internal.h"

namespace harp_fuse {

struct HostPhase {
    int t0, t1;          // stages [t0, t1)
    int B;               // fused block size
    int64_t S;           // natural stride of the phase (= s_{t0})
    int64_t W;           // shared-memory element stride of the phase's local index
    int lane_mult;       // 1, 2 or (B = 16 only) 4
};

inline uint16_t f2bf(double v) {
    const float f = (float)v;
    uint32_t u;
    std::memcpy(&u, &f, 4);
    const uint32_t r = u + 0x7FFFu + ((u >> 16) & 1u);
    return (uint16_t)(r >> 16);
}

// Fused block of phase hp for the block whose coordinates are base + r*S (r < B):
// F[r_in][r_out] in fp64, the product of the phase's stages restricted to those coordinates.
inline void fused_block(const harp_plan *plan, const HostPhase &hp, int64_t base, std::vector<double> &F) {
    const int B = hp.B;
    F.assign((size_t)B * B, 0.0);
    std::vector<double> before;
    for (int t = hp.t0; t < hp.t1; ++t) {
        const int b = plan->st.b[t];
        const int64_t s = plan->st.s[t];
        const int64_t ls = s / hp.S;                     // local stride of this stage's digit
        const float *Kt = plan->h_blocks.data() + plan->st.off[t];
        if (t > hp.t0) {
            before = F;
            std::fill(F.begin(), F.end(), 0.0);
        }
        for (int r = 0; r < B; ++r) {                    // r = output local index
            const int digit = (int)((r / ls) % b);
            const int r_base = r - digit * (int)ls;
            const int64_t pos = base + (int64_t)r_base * hp.S;      // coordinate with the digit zeroed
            const int64_t alpha = pos / ((int64_t)b * s), beta = pos % s;
            const float *Kc = Kt + (alpha * s + beta) * b * b;
            for (int i = 0; i < b; ++i) {                // input digit
                const int r_in = r_base + i * (int)ls;
                const double k = (double)Kc[i * b + digit];
                if (t == hp.t0) F[(size_t)r_in * B + r] = k;        // times the identity
                else
                    for (int row = 0; row < B; ++row) F[(size_t)row * B + r] += before[(size_t)row * B + r_in] * k;
            }
        }
    }
}

// slot maps: k-slot (or n-slot) index 0..B-1 of the MMA operand -> block-local index r
inline int strided_slot(int kappa, int B, int lane_mult) {
    const int qq = (kappa & 7) >> 1, i = kappa & 1, k = kappa >> 3;
    const int j = i + 2 * k;
    if (B == 16) {
        static const int joff1[4] = {0, 4, 8, 12}, joff2[4] = {0, 1, 8, 9}, joff4[4] = {0, 1, 2, 3};
        return lane_mult * qq + (lane_mult == 1 ? joff1[j] : lane_mult == 2 ? joff2[j] : joff4[j]);
    }
    static const int joff1[2] = {0, 4}, joff2[2] = {0, 1};
    return lane_mult * qq + (lane_mult == 1 ? joff1[j] : joff2[j]);
}

// a fused group of stages [t0, t1): operand width, real coordinates of a block, natural stride
struct GPhase {
    int t0, t1;
    int B, B_real;
    int64_t S;
};

// Fragment words of one block of a pass (mma.sync B operand, zero-padded), signs folded into the first stage:
// lane i's words (four for B = 16, one for B = 8) go to dst + i * lane_words.
template <typename Slot>
inline void block_fragment(const harp_plan *plan, const GPhase &gp, int64_t base, int dir, const Slot &slot, uint32_t *dst, int lane_words,
                           std::vector<double> &F) {
    const int Br = gp.B_real;
    fused_block(plan, HostPhase{gp.t0, gp.t1, Br, gp.S, 0, 1}, base, F);
    auto G = [&](int rin, int rout) -> double {
        if (rin >= Br || rout >= Br) return 0.0;
        double v = dir == 0 ? F[(size_t)rin * Br + rout] : F[(size_t)rout * Br + rin];
        if (gp.t0 == 0 && !plan->h_signs.empty()) {
            const int64_t pos = base + (int64_t)(dir == 0 ? rin : rout) * gp.S;
            v *= (double)plan->h_signs[(size_t)(plan->h_perm.empty() ? pos : plan->h_perm[(size_t)pos])];
        }
        return v;
    };
    for (int lane = 0; lane < 32; ++lane, dst += lane_words) {
        const int gg = lane >> 2, qq = lane & 3;
        for (int nt = 0; nt < gp.B / 8; ++nt) {
            const int n = slot(8 * nt + gg);
            for (int h = 0; h < gp.B / 8; ++h)
                dst[gp.B / 8 * nt + h] = f2bf(G(slot(8 * h + 2 * qq), n)) | ((uint32_t)f2bf(G(slot(8 * h + 2 * qq + 1), n)) << 16);
        }
    }
}

}  // namespace harp_fuse

// passes fed by the copy engine (harp_pipe.cu)
struct PipePlan;
// fragments of a pass that the plan already holds: [direction][column group][words], first words of the phases, slot maps
struct PassFrags {
    const uint32_t *bfrag[2];
    int32_t words, off[2][6], lm[6];
};
harp_status_t harp_pipe_build(const harp_plan *plan, const std::vector<harp_fuse::GPhase> &phs, bool lower, int64_t S_mid, int64_t U,
                              bool wide, const PassFrags &fr, PipePlan **out);
int64_t harp_pipe_min_rows(const PipePlan *pp);   // smallest batch that it is meant for
void harp_pipe_destroy(PipePlan *pp);
harp_status_t harp_pipe_apply(const PipePlan *pp, void *x, int64_t n_rows, int transpose, bool overlap, cudaStream_t stream);
int32_t harp_pipe_error_word(const PipePlan *pp);
