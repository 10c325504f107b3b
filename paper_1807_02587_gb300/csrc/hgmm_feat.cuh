// Canonical-frame features of a GMM tree for the learned pose proposal.
//
// Frame of a cloud: c = root mean, s = sqrt(trace Sigma_root) (RMS radius),
// V = the root eigenvectors in columns as the build computed them (the axes
// that seeded the level-0 children), third column negated when det V < 0 so
// that V is a rotation.  Features (64 nodes x 10, BF16): level-0 node k goes
// to group k ^ (4 if the third axis was negated), i.e. the octant of its
// initial mean in the frame; inside a group the live children follow in
// order of decreasing weight (ties by index), and a live level-0 node whose
// children all died stands for itself in the group's first slot.  Entry:
// [64 pi_parent pi_child, V^T (mu - c) / s, 16 upper(V^T Sigma V) / s^2];
// empty slots are zero.  Frame record (16 float64): c, s, V row-major,
// flipped, 0, 0.
#pragma once

#include <cuda_bf16.h>

#include "hgmm_internal.cuh"
#include "hgmm_math.cuh"

namespace hgmm {

constexpr int FEAT_NODES = 64;
constexpr int FEAT_PER_NODE = 10;
constexpr int FEAT_PER_CLOUD = FEAT_NODES * FEAT_PER_NODE;
constexpr int FRAME_DOUBLES = 16;

__device__ __forceinline__ void feat_entry(__nv_bfloat16* out, double w, const double* mu,
                                           const double* S, const double* fr) {
    const double rs = rcp_f64(fr[3]);  // one reciprocal for the four scalings
    const double* V = fr + 4;  // V[i * 3 + a]: component i of axis a
    const double d[3] = {mu[0] - fr[0], mu[1] - fr[1], mu[2] - fr[2]};
    const double Sf[3][3] = {{S[0], S[1], S[2]}, {S[1], S[3], S[4]}, {S[2], S[4], S[5]}};
    out[0] = __double2bfloat16(64.0 * w);
    for (int a = 0; a < 3; ++a)
        out[1 + a] = __double2bfloat16((V[a] * d[0] + V[3 + a] * d[1] + V[6 + a] * d[2]) * rs);
    // (V^T Sigma V)_ab, upper triangle xx xy xz yy yz zz
    double SV[3][3];
    for (int i = 0; i < 3; ++i)
        for (int b = 0; b < 3; ++b)
            SV[i][b] = Sf[i][0] * V[b] + Sf[i][1] * V[3 + b] + Sf[i][2] * V[6 + b];
    const int ua[6] = {0, 0, 0, 1, 1, 2}, ub[6] = {0, 1, 2, 1, 2, 2};
    const double k = 16.0 * (rs * rs);
    for (int e = 0; e < 6; ++e) {
        const int a = ua[e], b = ub[e];
        out[4 + e] = __double2bfloat16(k * (V[a] * SV[0][b] + V[3 + a] * SV[1][b] + V[6 + a] * SV[2][b]));
    }
}

// Run by NT threads (whole warps, threadIdx.x < NT), which meet at sync();
// fsm = 16 doubles of shared memory.  Writes the 640 features and, if frame
// is not NULL, the frame record.  One thread per level-1 node, its rank among
// its siblings by shuffles in their group of eight lanes (a tree's features
// took 41 us with one lane per level-0 node sorting and writing eight
// children; two trees take 8.9 us in one launch with 64 threads each).  The weights are positive, so their bit
// patterns order as the values do.
template <int NT, typename Sync>
__device__ __forceinline__ void tree_features(const RootDev* __restrict__ root, const NodeStat* __restrict__ stat,
                                              __nv_bfloat16* __restrict__ feat, double* __restrict__ frame,
                                              double* fsm, Sync sync) {
    static_assert(NT % 32 == 0 && FEAT_NODES % NT == 0, "whole warps, equal shares");
    if (threadIdx.x == 0) {
        double V[9];
        for (int v = 0; v < 9; ++v) V[v] = root->V[v];
        const double det = V[0] * (V[4] * V[8] - V[5] * V[7]) - V[1] * (V[3] * V[8] - V[5] * V[6]) +
                           V[2] * (V[3] * V[7] - V[4] * V[6]);
        const bool flip = det < 0.0;
        if (flip) {
            V[2] = -V[2];
            V[5] = -V[5];
            V[8] = -V[8];
        }
        const double t = fmax(root->lam[0], 0.0) + fmax(root->lam[1], 0.0) + fmax(root->lam[2], 0.0);
        const double s = t > 0.0 ? t * rsqrt_f64(t) : 1.0;
        for (int a = 0; a < 3; ++a) fsm[a] = root->mu[a];
        fsm[3] = s;
        for (int v = 0; v < 9; ++v) fsm[4 + v] = V[v];
        fsm[13] = flip ? 1.0 : 0.0;
        fsm[14] = 0.0;
        fsm[15] = 0.0;
    }
    for (int i = threadIdx.x; i < FEAT_PER_CLOUD / 2; i += NT)
        reinterpret_cast<__nv_bfloat162*>(feat)[i] = __floats2bfloat162_rn(0.f, 0.f);
    sync();
    if (frame && threadIdx.x < FRAME_DOUBLES) frame[threadIdx.x] = fsm[threadIdx.x];
#pragma unroll 1
    for (int n = threadIdx.x; n < FEAT_NODES; n += NT) {
        const int k = n >> 3, j = n & 7, lane = threadIdx.x & 31;
        const NodeStat& P = stat[k];
        const NodeStat& C = stat[8 + n];
        const bool live = C.live != 0;
        const long long w = live ? __double_as_longlong(C.pi) : -1;
        int rank = 0;
#pragma unroll
        for (int o = 0; o < 8; ++o) {
            const long long x = __shfl_sync(0xffffffffu, w, (lane & 24) + o);
            rank += x > w || (x == w && o < j);
        }
        const bool any = __any_sync(0xffu << (lane & 24), live);
        const int group = k ^ (fsm[13] != 0.0 ? 4 : 0);
        // a live parent without live children stands in its group's first slot
        const bool self = !any && j == 0;
        if (P.live && (live || self)) {
            const NodeStat& N = live ? C : P;
            feat_entry(feat + (group * 8 + (live ? rank : 0)) * FEAT_PER_NODE, live ? P.pi * C.pi : P.pi, N.mu, N.S,
                       fsm);
        }
    }
    sync();
}

}  // namespace hgmm
