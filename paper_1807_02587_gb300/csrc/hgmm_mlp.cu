// Learned pose proposal: the network's forward and backward passes on the
// tensor cores (hgmm_tc.cuh), its loss through the 6-D rotation
// representation, Adam, the canonical-frame features of a tree, and the
// pose encode / decode / fallback-select kernels.
//
// Forward (x: batch x 1280 BF16):
//   H1 = relu(x W1^T + b1)      tcgen05, N = 256, K = 1280, bias+ReLU epilogue -> BF16
//   H2 = relu(H1 W2^T + b2)     tcgen05, N = 256, K = 256
//   Y  = H2 W3^T + b3           tcgen05, N = 16 (rows 9..15 of W3 are zero), FP32 out
// Backward (hgmm_train.cuh; dY from the loss kernel, BF16 for the tensor cores, FP32 kept):
//   dZ2 = (dY W3) * [H2 > 0], dZ1 = (dZ2 W2) * [H1 > 0]   one launch per 128-row block
//   dW3^T = H2^T dY, dW2 = dZ2^T H1, dW1 = dZ1^T x        one launch, operands read transposed
//   db = column sums of dZ1, dZ2, dY (two-pass, fixed order: deterministic)
//   K slices summed in order, with Adam in the same pass
#include <cuda_bf16.h>
#include <cudaTypedefs.h>
#include <mutex>

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <vector>

#include "../../include/hgmm_proposal.h"
#include "hgmm_feat.cuh"
#include "hgmm_internal.cuh"
#include "hgmm_math.cuh"
#include "hgmm_tc.cuh"

namespace hgmm {
namespace {

constexpr int IN = HGMM_MLP_IN, HID = HGMM_MLP_HIDDEN, OUT = HGMM_MLP_OUT, OUTP = 16;
constexpr int64_t OFF_W1 = 0;
constexpr int64_t OFF_B1 = OFF_W1 + int64_t(HID) * IN;
constexpr int64_t OFF_W2 = OFF_B1 + HID;
constexpr int64_t OFF_B2 = OFF_W2 + int64_t(HID) * HID;
constexpr int64_t OFF_W3 = OFF_B2 + HID;
constexpr int64_t OFF_B3 = OFF_W3 + int64_t(OUT) * HID;
constexpr int64_t N_PARAMS = OFF_B3 + OUT;
static_assert(N_PARAMS == HGMM_MLP_PARAMS, "parameter layout");
static_assert(FEAT_PER_CLOUD == HGMM_FEAT_PER_CLOUD && FRAME_DOUBLES == HGMM_FRAME_DOUBLES, "layout");

constexpr int ERR_TIMEOUT = 1;
constexpr int ERR_INDEX = 2;
constexpr int COLSUM_ROWS = 64;  // rows per partial column sum

using bf16 = __nv_bfloat16;

// Features and frames of one or two trees (blockIdx.x), one thread per node.
struct FeatJob {
    const RootDev* root;
    const NodeStat* stat;
    bf16* feat;
    double* frame;
};

__global__ void __launch_bounds__(FEAT_NODES) k_tree_features(FeatJob a, FeatJob b) {
    __shared__ double fsm[FRAME_DOUBLES];
    const FeatJob j = blockIdx.x == 0 ? a : b;
    tree_features<FEAT_NODES>(j.root, j.stat, j.feat, j.frame, fsm, [] { __syncthreads(); });
}

// Rows idx[r] of x and labels -> row r of the gathered batch.
__global__ void k_gather(const bf16* __restrict__ X, const float* __restrict__ L,
                         const int* __restrict__ idx, int n_rows, bf16* __restrict__ Xo,
                         float* __restrict__ Lo, int* __restrict__ err) {
    const int r = blockIdx.x;
    const int src = idx[r];
    const bool good = src >= 0 && src < n_rows;
    if (!good && threadIdx.x == 0) atomicOr(err, ERR_INDEX);
    const uint4* xs = reinterpret_cast<const uint4*>(X + int64_t(good ? src : 0) * IN);
    uint4* xd = reinterpret_cast<uint4*>(Xo + int64_t(r) * IN);
    for (int i = threadIdx.x; i < IN / 8; i += blockDim.x)
        xd[i] = good ? __ldg(xs + i) : make_uint4(0u, 0u, 0u, 0u);
    if (threadIdx.x < HGMM_LABEL_FLOATS)
        Lo[int64_t(r) * HGMM_LABEL_FLOATS + threadIdx.x] =
            good ? L[int64_t(src) * HGMM_LABEL_FLOATS + threadIdx.x] : 0.f;
}

__device__ __forceinline__ void cross3(const double* a, const double* b, double* c) {
    c[0] = a[1] * b[2] - a[2] * b[1];
    c[1] = a[2] * b[0] - a[0] * b[2];
    c[2] = a[0] * b[1] - a[1] * b[0];
}
__device__ __forceinline__ double dot3(const double* a, const double* b) {
    return a[0] * b[0] + a[1] * b[1] + a[2] * b[2];
}

__device__ __forceinline__ void load_frame(const double* f, double* c, double& s, double* V) {
    for (int a = 0; a < 3; ++a) c[a] = f[a];
    s = f[3];
    for (int v = 0; v < 9; ++v) V[v] = f[4 + v];
}

// Gram-Schmidt of a network output's first six values into the columns b1, b2,
// b3 = b1 x b2 of R'.
__device__ __forceinline__ void decode_basis(const float* y, double* b1, double* b2, double* b3) {
    double a1[3], a2[3], u[3];
    for (int k = 0; k < 3; ++k) {
        a1[k] = y[k];
        a2[k] = y[3 + k];
    }
    const double s1 = dot3(a1, a1);
    const double i1 = s1 > 0.0 ? rsqrt_f64(s1) : 0.0;
    for (int k = 0; k < 3; ++k) b1[k] = a1[k] * i1;
    const double dd = dot3(b1, a2);
    for (int k = 0; k < 3; ++k) u[k] = a2[k] - dd * b1[k];
    const double s2 = dot3(u, u);
    const double i2 = s2 > 0.0 ? rsqrt_f64(s2) : 0.0;
    for (int k = 0; k < 3; ++k) b2[k] = u[k] * i2;
    cross3(b1, b2, b3);
}

// Sixteen lanes per pair, lane (r, c) = entry (r, c) of T: a handful of pairs
// is one dependent FP64 chain, so the entries share its instructions (one
// pair: 6.8 us with one thread, 4.6 here).  The chain before the entries is
// run sixteen times over, so from a few thousand pairs on, where the FP64 pipes
// are busy, k_decode_many's one thread per pair is faster: calls of 4,096 /
// 8,192 / 65,536 pairs take 12.8 / 21 / 118 us here, 9.5 / 9.5 / 24 there; at
// 2,048 both take the 9.2 of the launch.
constexpr int DECODE_THREADS = 128;
constexpr int DECODE_FEW = 2048;
__global__ void __launch_bounds__(DECODE_THREADS)
k_decode(const float* __restrict__ Y, const double* __restrict__ F, int n, double* __restrict__ T) {
    const int64_t i = (int64_t(blockIdx.x) * DECODE_THREADS + threadIdx.x) >> 4;
    const unsigned half = 0xFFFFu << (threadIdx.x & 16);
    if (i >= n) return;  // whole half-warps
    const int e = threadIdx.x & 15, r = e >> 2 < 3 ? e >> 2 : 2, c = e & 3;
    double cs[3], ct[3], Vs[9], Vt[9], ss, st;
    load_frame(F + 32 * i, cs, ss, Vs);
    load_frame(F + 32 * i + 16, ct, st, Vt);
    const float* y = Y + i * OUT;
    double b1[3], b2[3], b3[3];
    decode_basis(y, b1, b2, b3);
    // R' (columns b1..b3); A = Vt R', R = A Vs^T: lane (r, c) forms entry (r,
    // c) of both; lane (r, 3) the translation's Vt y_t instead of A's entry
    const double vt0 = r == 0 ? Vt[0] : (r == 1 ? Vt[3] : Vt[6]);
    const double vt1 = r == 0 ? Vt[1] : (r == 1 ? Vt[4] : Vt[7]);
    const double vt2 = r == 0 ? Vt[2] : (r == 1 ? Vt[5] : Vt[8]);
    double x[3];
    for (int k = 0; k < 3; ++k) x[k] = c == 0 ? b1[k] : (c == 1 ? b2[k] : (c == 2 ? b3[k] : double(y[6 + k])));
    const double Arc = vt0 * x[0] + vt1 * x[1] + vt2 * x[2];
    const int row = threadIdx.x & 28;  // this lane's row of four
    const double A0 = __shfl_sync(half, Arc, row & 31), A1 = __shfl_sync(half, Arc, (row + 1) & 31);
    const double A2 = __shfl_sync(half, Arc, (row + 2) & 31);
    double z[3];
    for (int k = 0; k < 3; ++k) z[k] = c == 1 ? Vs[3 + k] : (c == 2 ? Vs[6 + k] : Vs[k]);
    const double Rrc = A0 * z[0] + A1 * z[1] + A2 * z[2];
    const double R0 = __shfl_sync(half, Rrc, row), R1 = __shfl_sync(half, Rrc, row + 1);
    const double R2 = __shfl_sync(half, Rrc, row + 2);
    const double ctr = r == 0 ? ct[0] : (r == 1 ? ct[1] : ct[2]);
    const double t = ctr + st * Arc - (R0 * cs[0] + R1 * cs[1] + R2 * cs[2]);
    T[16 * i + e] = e >= 12 ? (e == 15 ? 1.0 : 0.0) : (c == 3 ? t : Rrc);
}

// The same, one thread per pair.
__global__ void __launch_bounds__(DECODE_THREADS)
k_decode_many(const float* __restrict__ Y, const double* __restrict__ F, int n, double* __restrict__ T) {
    const int64_t i = int64_t(blockIdx.x) * DECODE_THREADS + threadIdx.x;
    if (i >= n) return;
    double cs[3], ct[3], Vs[9], Vt[9], ss, st, b[3][3];
    load_frame(F + 32 * i, cs, ss, Vs);
    load_frame(F + 32 * i + 16, ct, st, Vt);
    const float* y = Y + i * OUT;
    decode_basis(y, b[0], b[1], b[2]);
    double* o = T + 16 * i;
    for (int r = 0; r < 3; ++r) {
        double A[3], R[3];
        for (int c = 0; c < 3; ++c) A[c] = Vt[3 * r] * b[c][0] + Vt[3 * r + 1] * b[c][1] + Vt[3 * r + 2] * b[c][2];
        for (int c = 0; c < 3; ++c) R[c] = A[0] * Vs[3 * c] + A[1] * Vs[3 * c + 1] + A[2] * Vs[3 * c + 2];
        const double vt = Vt[3 * r] * y[6] + Vt[3 * r + 1] * y[7] + Vt[3 * r + 2] * y[8];
        for (int c = 0; c < 3; ++c) o[4 * r + c] = R[c];
        o[4 * r + 3] = ct[r] + st * vt - (R[0] * cs[0] + R[1] * cs[1] + R[2] * cs[2]);
    }
    for (int c = 0; c < 4; ++c) o[12 + c] = c == 3 ? 1.0 : 0.0;
}

__global__ void k_encode(const double* __restrict__ T, const double* __restrict__ F, int n,
                         float* __restrict__ L) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    double cs[3], ct[3], Vs[9], Vt[9], ss, st;
    load_frame(F + 32 * int64_t(i), cs, ss, Vs);
    load_frame(F + 32 * int64_t(i) + 16, ct, st, Vt);
    const double* p = T + 16 * int64_t(i);
    double RVs[3][3];
    for (int r = 0; r < 3; ++r)
        for (int c = 0; c < 3; ++c)
            RVs[r][c] = p[4 * r] * Vs[c] + p[4 * r + 1] * Vs[3 + c] + p[4 * r + 2] * Vs[6 + c];
    float* l = L + int64_t(i) * HGMM_LABEL_FLOATS;
    for (int r = 0; r < 3; ++r)
        for (int c = 0; c < 3; ++c)
            l[3 * r + c] = float(Vt[r] * RVs[0][c] + Vt[3 + r] * RVs[1][c] + Vt[6 + r] * RVs[2][c]);
    double d[3];
    for (int r = 0; r < 3; ++r)
        d[r] = p[4 * r] * cs[0] + p[4 * r + 1] * cs[1] + p[4 * r + 2] * cs[2] + p[4 * r + 3] - ct[r];
    for (int a = 0; a < 3; ++a) l[9 + a] = float((Vt[a] * d[0] + Vt[3 + a] * d[1] + Vt[6 + a] * d[2]) / st);
}

// One thread per pair; inputs and outputs may alias (T_out = T_a, obj_out
// = obj_a): every value is read before it is written.
__global__ void k_select(int n, const double* Ta, const double* oa, const double* Tb, const double* ob,
                         double* To, int* __restrict__ choice, double* oo) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double a = oa[i], b = ob[i];
    const bool take_b = isfinite(b) && (!isfinite(a) || b < a);
    const double* src = (take_b ? Tb : Ta) + 16 * int64_t(i);
    double v[16];
    for (int k = 0; k < 16; ++k) v[k] = src[k];
    for (int k = 0; k < 16; ++k) To[16 * int64_t(i) + k] = v[k];
    if (choice) choice[i] = take_b ? 1 : 0;
    if (oo) oo[i] = take_b ? b : a;
}

__global__ void k_compose(int n, const double* __restrict__ A, const double* __restrict__ Bm,
                          double* __restrict__ O) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double* a = A + 16 * int64_t(i);
    const double* b = Bm + 16 * int64_t(i);
    double* o = O + 16 * int64_t(i);
    for (int r = 0; r < 4; ++r)
        for (int c = 0; c < 4; ++c)
            o[4 * r + c] = a[4 * r] * b[c] + a[4 * r + 1] * b[4 + c] + a[4 * r + 2] * b[8 + c] + a[4 * r + 3] * b[12 + c];
}


// ---------------------------------------------------------------------------
// The whole forward pass of one 128-row block in one launch (warp-specialised
// tcgen05 with TMEM accumulators and TMA operand streams):
//   layer 1: acc1 (TMEM columns 0..255) = X[128 x 1280] W1^T, 20 K-steps of
//            TMA-fed 128 x 64 / 256 x 64 tiles in a 4-stage ring;
//   epilogue warps: h1 = relu(acc1 + b1) as BF16 into shared memory in the
//            128-byte-swizzled K-major layout that TMA would write, as layer 2's
//            A operand, one 64-column chunk after the other: layer 2's products
//            of a chunk start when it is there;
//   layer 2: acc2 (columns 256..511) = h1 W2^T, W2 tiles streamed by TMA;
//   epilogue: h2 likewise (over h1);
//   layer 3: acc3 (columns 0..15) = h2 W3^T (W3 padded to 16 rows);
//   epilogue: Y = acc3 + b3 (9 columns, FP32).
// For the backward pass the chunks also go to H1 and H2 by TMA stores.
// Warps 0-7 are the epilogue (warp w owns TMEM lanes 32 (w mod 4)..., i.e.
// rows, and half w / 4 of a chunk's columns), one thread of warp 8 issues the
// TMA loads, warp 9 the MMAs.  Every wait is bounded; on a timeout the kernel
// records the error, lets every role run out (commits and arrivals still
// happen) and drains its loads in flight before it frees TMEM.
// A block is a chain on one SM: 20 K steps of four 128 x 256 x 16 MMAs at the
// tensor pipe's own rate (0.385 us each, 7.7 us in all), then two epilogues and
// layers: 18.9 us per call from 1 to 9,728 rows with four epilogue warps and
// whole-layer hand-overs, 15.7 to 16.5 now; 16,384 rows (128 blocks) 20.7 against
// 16.8.  Splitting a block's columns over a cluster of two or
// four CTAs does not shorten it: an MMA of 128 or 64 columns takes 0.075 us
// against 0.096 for 256, and handing the hidden layers round through
// distributed shared memory costs more than the shorter epilogues save (20.9 us
// against 18.9 per call at 8192 rows, 17.3 against 18.8 at one row).
constexpr int FW_THREADS = 320;
constexpr int FW_S1 = 4;                          // layer-1 stages
constexpr int FW_A = 128 * 128;                   // 128 rows x 64 BF16
constexpr int FW_B = 256 * 128;                   // 256 rows x 64 BF16
constexpr int FW_STAGE1 = FW_A + FW_B;            // 48 KB
constexpr int FW_H = 4 * FW_A;                    // 128 x 256 BF16: four 64-wide K chunks (64 KB)
constexpr int FW_W2_OFF = FW_H;                   // two 32 KB W2 stages after the h buffer
constexpr int FW_W3_OFF = FW_W2_OFF + 2 * FW_B;   // four 16 x 64 W3 tiles (8 KB)
constexpr int FW_W3_TILE = 16 * 128;
constexpr int FW_SMEM = FW_S1 * FW_STAGE1 + 1024; // the h buffer and W2/W3 reuse the layer-1 ring
static_assert(FW_W3_OFF + 4 * FW_W3_TILE <= FW_S1 * FW_STAGE1, "layer 2/3 buffers inside the ring");

// Row r's 16-byte unit u of a 64-wide K chunk in the 128-byte swizzled layout.
__device__ __forceinline__ uint32_t sw128_offset(int r, int u) {
    return uint32_t(r * 128 + ((u ^ (r & 7)) << 4));
}

// relu(acc + bias) of this thread's row and one half (32 columns) of a
// 64-column chunk, as BF16 into the chunk's swizzled tile.
__device__ __forceinline__ void fw_hidden_epilogue(uint32_t tacc, const float* __restrict__ bias, uint32_t chunk,
                                                   int r, int half) {
    float v[32];
    tc::tmem_ld32(tacc, v);
    const float4* b4 = reinterpret_cast<const float4*>(bias);
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const float4 ba = __ldg(b4 + 2 * u), bb = __ldg(b4 + 2 * u + 1);
        const float x[8] = {v[8 * u] + ba.x, v[8 * u + 1] + ba.y, v[8 * u + 2] + ba.z, v[8 * u + 3] + ba.w,
                            v[8 * u + 4] + bb.x, v[8 * u + 5] + bb.y, v[8 * u + 6] + bb.z, v[8 * u + 7] + bb.w};
        uint32_t w[4];
#pragma unroll
        for (int h = 0; h < 4; ++h) {
            const __nv_bfloat162 p2 = __floats2bfloat162_rn(fmaxf(x[2 * h], 0.f), fmaxf(x[2 * h + 1], 0.f));
            w[h] = *reinterpret_cast<const uint32_t*>(&p2);
        }
        asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};"
                     :: "r"(chunk + sw128_offset(r, 4 * half + u)), "r"(w[0]), "r"(w[1]), "r"(w[2]), "r"(w[3])
                     : "memory");
    }
}

// The four K = 16 steps of a 64-wide K chunk by a converged warp (32 bytes
// along the swizzled row per step: the descriptors' address field counts 16
// bytes), and a commit on bar if it is not null.
__device__ __forceinline__ void mma_k64(bool lead, uint32_t tmem, uint64_t da, uint64_t db, uint32_t idesc,
                                        bool accumulate, uint64_t* bar) {
    if (lead) {
#pragma unroll
        for (int kk = 0; kk < 4; ++kk)
            tc::mma_bf16(tmem, da + 2 * kk, db + 2 * kk, idesc, accumulate || kk != 0 ? 1u : 0u);
        if (bar) tc::mma_commit(bar);
    }
    __syncwarp();
}

__device__ __forceinline__ void tma_store_2d(const void* tmap, int x, int y, uint32_t src) {
    asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%1, %2}], [%3];"
                 :: "l"(tmap), "r"(x), "r"(y), "r"(src) : "memory");
}
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_read() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }

__device__ __forceinline__ bool fw_wait(uint64_t* bar, uint32_t parity, int* fail) {
    if (*(volatile int*)fail) return false;
    if (tc::mbar_wait_bounded(bar, parity, tc::MBAR_SPIN_LIMIT)) return true;
    atomicExch(fail, 1);
    return false;
}

__global__ void __launch_bounds__(FW_THREADS, 1)
k_mlp_forward(const __grid_constant__ CUtensorMap tmX, const __grid_constant__ CUtensorMap tmW1,
              const __grid_constant__ CUtensorMap tmW2, const __grid_constant__ CUtensorMap tmW3,
              const __grid_constant__ CUtensorMap tmH1, const __grid_constant__ CUtensorMap tmH2,
              const float* __restrict__ b1, const float* __restrict__ b2, const float* __restrict__ b3p,
              bool keep_hidden, float* __restrict__ Y, int batch, int* __restrict__ err) {
    extern __shared__ unsigned char fw_raw[];
    __shared__ __align__(8) uint64_t full1[FW_S1], empty1[FW_S1], full2[2], empty2[2];
    __shared__ __align__(8) uint64_t full3, done1, done2, done3, h1_ready[4], h2_ready[4];
    __shared__ uint32_t tmem_slot;
    __shared__ int fail;
    const uint32_t base = (tc::smem_u32(fw_raw) + 1023u) & ~1023u;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int m0 = blockIdx.x * 128;
    constexpr int NK1 = IN / 64, NK2 = HID / 64;
    constexpr uint32_t ID1 = tc::idesc_bf16_f32(128, HID), ID3 = tc::idesc_bf16_f32(128, OUTP);
    if (warp == 8) {
        tc::tmem_alloc(&tmem_slot, 512);
        tc::tmem_relinquish();
    }
    if (threadIdx.x == 288) {
        for (int i = 0; i < FW_S1; ++i) {
            tc::mbar_init(&full1[i], 1);
            tc::mbar_init(&empty1[i], 1);
        }
        for (int i = 0; i < 2; ++i) {
            tc::mbar_init(&full2[i], 1);
            tc::mbar_init(&empty2[i], 1);
        }
        tc::mbar_init(&full3, 1);
        tc::mbar_init(&done1, 1);
        tc::mbar_init(&done2, 1);
        tc::mbar_init(&done3, 1);
        for (int i = 0; i < 4; ++i) {
            tc::mbar_init(&h1_ready[i], 256);
            tc::mbar_init(&h2_ready[i], 256);
        }
        fail = 0;
        tc::fence_mbar_init();
        tc::prefetch_tmap(&tmX);
        tc::prefetch_tmap(&tmW1);
        tc::prefetch_tmap(&tmW2);
        tc::prefetch_tmap(&tmW3);
    }
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t tmem = tmem_slot;
    const uint32_t hbuf = base;
    int issued1 = 0, issued2 = 0;
    bool issued3 = false;
    if (threadIdx.x == 256) {
        // ---- producer
        for (int kt = 0; kt < NK1; ++kt) {
            const int st = kt % FW_S1;
            if (kt >= FW_S1 && !fw_wait(&empty1[st], ((kt / FW_S1) - 1) & 1, &fail)) break;
            const uint32_t sa = base + st * FW_STAGE1;
            tc::mbar_arrive_expect_tx(&full1[st], uint32_t(FW_STAGE1));
            tc::tma_load_2d(sa, &tmX, kt * 64, m0, &full1[st]);
            tc::tma_load_2d(sa + FW_A, &tmW1, kt * 64, 0, &full1[st]);
            issued1 = kt + 1;
        }
        // layer 2 and 3 operands go where the layer-1 ring was: after its MMAs
        if (issued1 == NK1 && fw_wait(&done1, 0, &fail)) {
            tc::mbar_arrive_expect_tx(&full3, uint32_t(4 * FW_W3_TILE));
            for (int kt = 0; kt < NK2; ++kt)
                tc::tma_load_2d(base + FW_W3_OFF + kt * FW_W3_TILE, &tmW3, kt * 64, 0, &full3);
            issued3 = true;
            for (int kt = 0; kt < NK2; ++kt) {
                const int st = kt & 1;
                if (kt >= 2 && !fw_wait(&empty2[st], ((kt >> 1) - 1) & 1, &fail)) break;
                tc::mbar_arrive_expect_tx(&full2[st], uint32_t(FW_B));
                tc::tma_load_2d(base + FW_W2_OFF + st * FW_B, &tmW2, kt * 64, 0, &full2[st]);
                issued2 = kt + 1;
            }
        }
    } else if (warp == 9) {
        // ---- MMA issuer: the warp runs converged, one lane issues (the
        // descriptors are then warp-uniform values)
        const bool lead = tc::elect_one();
        bool ok = true;
        for (int kt = 0; kt < NK1 && ok; ++kt) {
            const int st = kt % FW_S1;
            ok = __all_sync(0xffffffffu, fw_wait(&full1[st], (kt / FW_S1) & 1, &fail));
            if (!ok) break;
            tc::fence_after_sync();
            const uint32_t sa = base + st * FW_STAGE1;
            mma_k64(lead, tmem, tc::smem_desc_sw128(sa), tc::smem_desc_sw128(sa + FW_A), ID1, kt != 0, &empty1[st]);
        }
        if (lead) tc::mma_commit(&done1);
        for (int kt = 0; kt < NK2 && ok; ++kt) {
            const int st = kt & 1;
            ok = __all_sync(0xffffffffu, fw_wait(&h1_ready[kt], 0, &fail) && fw_wait(&full2[st], (kt >> 1) & 1, &fail));
            if (!ok) break;
            tc::fence_after_sync();
            mma_k64(lead, tmem + 256u, tc::smem_desc_sw128(hbuf + kt * FW_A),
                    tc::smem_desc_sw128(base + FW_W2_OFF + st * FW_B), ID1, kt != 0, &empty2[st]);
            if (lead && keep_hidden) {
                tma_store_2d(&tmH1, kt * 64, m0, hbuf + kt * FW_A);
                bulk_commit();
            }
        }
        if (lead) {
            bulk_wait_read();  // h1 has left the buffer that h2 takes after done2
            tc::mma_commit(&done2);
        }
        ok = ok && __all_sync(0xffffffffu, fw_wait(&full3, 0, &fail));
        for (int kt = 0; kt < NK2 && ok; ++kt) {
            ok = __all_sync(0xffffffffu, fw_wait(&h2_ready[kt], 0, &fail));
            if (!ok) break;
            tc::fence_after_sync();
            mma_k64(lead, tmem, tc::smem_desc_sw128(hbuf + kt * FW_A),
                    tc::smem_desc_sw128(base + FW_W3_OFF + kt * FW_W3_TILE), ID3, kt != 0, nullptr);
            if (lead && keep_hidden) {
                tma_store_2d(&tmH2, kt * 64, m0, hbuf + kt * FW_A);
                bulk_commit();
            }
        }
        if (lead) {
            tc::mma_commit(&done3);
            bulk_wait();
        }
    } else if (warp < 8) {
        // ---- epilogue: thread = tile row and half of every chunk
        const int r = (warp & 3) * 32 + lane, half = warp >> 2;
        const int m = m0 + r;
        const uint32_t lanes = uint32_t((warp & 3) * 32) << 16;
        auto hidden = [&](bool ok, uint32_t acc, const float* bias, uint64_t* ready) {
            if (ok) tc::fence_after_sync();
#pragma unroll 1
            for (int c = 0; c < NK2; ++c) {
                if (ok) {
                    fw_hidden_epilogue(tmem + lanes + acc + uint32_t(64 * c + 32 * half), bias + 64 * c + 32 * half,
                                       hbuf + uint32_t(c * FW_A), r, half);
                    tc::fence_before_sync();
                }
                tc::fence_proxy_async();  // the chunk, written here, is read by the tensor core and by TMA
                asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" :: "r"(tc::smem_u32(ready + c)) : "memory");
            }
        };
        // warp-uniform decisions: the TMEM loads are warp-collective
        const bool ok1 = __all_sync(0xffffffffu, fw_wait(&done1, 0, &fail));
        hidden(ok1, 0u, b1, h1_ready);
        const bool ok2 = __all_sync(0xffffffffu, ok1 && fw_wait(&done2, 0, &fail));
        hidden(ok2, 256u, b2, h2_ready);
        if (warp < 4) {
            const bool ok3 = __all_sync(0xffffffffu, ok2 && fw_wait(&done3, 0, &fail));
            if (ok3) {
                tc::fence_after_sync();
                float v[16];
                tc::tmem_ld16(tmem + lanes, v);
                if (m < batch)
#pragma unroll
                    for (int j = 0; j < OUT; ++j) Y[int64_t(m) * OUT + j] = v[j] + b3p[j];
            }
        }
    }
    __syncwarp();
    if (threadIdx.x == 256) {
        // loads issued but never consumed: let them land before the CTA exits
        for (int kt = max(0, issued1 - FW_S1); kt < issued1; ++kt)
            tc::mbar_wait_bounded(&full1[kt % FW_S1], (kt / FW_S1) & 1, tc::MBAR_SPIN_LIMIT);
        for (int kt = max(0, issued2 - 2); kt < issued2; ++kt)
            tc::mbar_wait_bounded(&full2[kt & 1], (kt >> 1) & 1, tc::MBAR_SPIN_LIMIT);
        if (issued3) tc::mbar_wait_bounded(&full3, 0, tc::MBAR_SPIN_LIMIT);
    }
    if (threadIdx.x == 288) tc::mbar_wait_bounded(&done3, 0, tc::MBAR_SPIN_LIMIT);  // MMAs in flight
    __syncthreads();
    if (threadIdx.x == 0 && *(volatile int*)&fail) atomicOr(err, ERR_TIMEOUT);
    tc::fence_before_sync();
    __syncthreads();
    if (warp == 8) tc::tmem_dealloc(tmem, 512);
}

}  // namespace
}  // namespace hgmm

#include "hgmm_train.cuh"

using namespace hgmm;
using hgmm::tc::GemmArgs;

struct hgmm_mlp {
    int device = 0;
    int max_batch = 0;
    int step = 0;
    std::vector<void*> allocs;
    float* P = nullptr;   // FP32 master parameters
    float* G = nullptr;   // gradients
    float* Mo = nullptr;  // Adam moments
    float* Vo = nullptr;
    bf16* W1 = nullptr;
    bf16* W2 = nullptr;
    bf16* W3 = nullptr;   // 16 x 256, rows >= 9 zero
    float* b3p = nullptr; // 16
    bf16* W2T = nullptr;  // W2 transposed (the backward pass)
    bf16* W3T = nullptr;  // W3 transposed, 256 x 64, columns >= 9 zero
    bf16* Xg = nullptr;   // gathered batch
    float* Lg = nullptr;
    bf16* H1 = nullptr;
    bf16* H2 = nullptr;
    float* Y = nullptr;   // batch x 9
    bf16* dY = nullptr;   // batch x 64, columns >= 9 zero
    float* dYf = nullptr;
    bf16* dZ2 = nullptr;
    bf16* dZ1 = nullptr;
    float* part = nullptr;
    float* loss = nullptr;
    double* loss_part = nullptr;  // per CTA of the loss
    unsigned* loss_cnt = nullptr;
    int* err = nullptr;
    float* ws = nullptr;      // K-slice partials of the weight gradients
    long long ws_cap = 0;     // floats
    bool maps = true;         // tensor maps may be used (checking aid: hgmm_debug_mlp_maps)
    bf16* prop_x = nullptr;   // hgmm_propose: one pair's input (1280)
    double* prop_fr = nullptr;  // ... its frames (source, target: 32)
    float* prop_y = nullptr;  // ... the network's output (9)
};

namespace {

template <typename T>
bool malloc_into(hgmm_mlp* m, T** p, size_t count) {
    *p = nullptr;
    if (cudaMalloc(reinterpret_cast<void**>(p), (count ? count : 1) * sizeof(T)) != cudaSuccess) return false;
    m->allocs.push_back(*p);
    return cudaMemset(*p, 0, (count ? count : 1) * sizeof(T)) == cudaSuccess;
}

bool a16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

// Operand (rows x K) at base with element strides (rs, ks): the tile loader
// needs 16-byte vectors along K (ks == 1) or along the rows (rs == 1).
bool operand_ok(const void* base, long long rs, long long ks, int rows, int K) {
    if (!a16(base)) return false;
    if (ks == 1) return rs % 8 == 0 && K % 8 == 0;
    if (rs == 1) return ks % 8 == 0 && rows % 8 == 0;
    return false;
}

constexpr int MAX_SLICES = 32;

template <int BN>
int gemm_launch(const GemmArgs& g, int slices, cudaStream_t s) {
    const dim3 grid((g.M + tc::GEMM_BM - 1) / tc::GEMM_BM, (g.N + BN - 1) / BN, slices);
    tc::k_gemm_bf16<BN><<<grid, tc::GEMM_THREADS, tc::gemm_smem_bytes(BN), s>>>(g);
    return cudaGetLastError() == cudaSuccess ? HGMM_OK : HGMM_ECUDA;
}

// cuTensorMapEncodeTiled from the driver (resolved once), or null.
PFN_cuTensorMapEncodeTiled_v12000 tmap_encoder() {
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
        else
            cudaGetLastError();
    });
    return fn;
}

// Tensor map of a K-contiguous BF16 operand (rows x K, row stride rs
// elements): dimensions (K, rows), box 64 x box_rows, 128-byte swizzle,
// zeros outside the matrix.
bool encode_operand(CUtensorMap* tm, const bf16* base, long long rs, int rows, int K, int box_rows) {
    PFN_cuTensorMapEncodeTiled_v12000 enc = tmap_encoder();
    if (!enc) return false;
    const cuuint64_t dims[2] = {cuuint64_t(K), cuuint64_t(rows)};
    const cuuint64_t strides[1] = {cuuint64_t(rs) * sizeof(bf16)};
    const cuuint32_t box[2] = {cuuint32_t(tc::GEMM_BK), cuuint32_t(box_rows)};
    const cuuint32_t estr[2] = {1, 1};
    return enc(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<bf16*>(base), dims, strides, box, estr,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <int BN>
int gemm_tma_launch(const GemmArgs& g, const CUtensorMap& ta, const CUtensorMap& tb, cudaStream_t s) {
    const dim3 grid((g.M + tc::GEMM_BM - 1) / tc::GEMM_BM, (g.N + BN - 1) / BN);
    tc::k_gemm_tma<BN><<<grid, tc::GEMM_THREADS, tc::tma_smem_bytes(BN), s>>>(ta, tb, g);
    return cudaGetLastError() == cudaSuccess ? HGMM_OK : HGMM_ECUDA;
}

// D = A B^T with the fused epilogue of g.  Both operands K-contiguous and
// no K slices: the warp-specialised TMA kernel.  Otherwise the cp.async
// kernel: N <= 16 runs 128 x 16 tiles, larger N 128 x 128 tiles; when the
// tiles alone cannot fill the GPU, K is long and there is a workspace (the
// weight gradients: K = batch), K is cut into 64-multiple slices whose FP32
// partials go to ws and are summed in a fixed order.  maps: tensor maps may be
// used.
int gemm(GemmArgs g, cudaStream_t s, float* ws = nullptr, long long ws_cap = 0, bool maps = true) {
    if (g.M < 1 || g.N < 1 || g.K < 1 || !operand_ok(g.A, g.a_m, g.a_k, g.M, g.K) ||
        !operand_ok(g.B, g.b_n, g.b_k, g.N, g.K))
        return HGMM_EINVAL;
    const int bn = g.N <= 16 ? 16 : 128;
    const int tiles = ((g.M + tc::GEMM_BM - 1) / tc::GEMM_BM) * ((g.N + bn - 1) / bn);
    const int kt = (g.K + tc::GEMM_BK - 1) / tc::GEMM_BK;
    int slices = 1;
    if (ws && g.epi == tc::EPI_F32 && tiles < 128) slices = std::min(std::min(MAX_SLICES, kt), (304 + tiles - 1) / tiles);
    g.k_split = ((kt + slices - 1) / slices) * tc::GEMM_BK;
    slices = (g.K + g.k_split - 1) / g.k_split;
    if (maps && slices <= 1 && g.a_k == 1 && g.b_k == 1) {
        // (operand_ok has checked 16-byte bases and row strides % 8 == 0)
        CUtensorMap ta, tb;
        if (encode_operand(&ta, g.A, g.a_m, g.M, g.K, tc::GEMM_BM) &&
            encode_operand(&tb, g.B, g.b_n, g.N, g.K, bn)) {
            g.k_split = g.K;
            g.split_stride = 0;
            return bn == 16 ? gemm_tma_launch<16>(g, ta, tb, s) : gemm_tma_launch<128>(g, ta, tb, s);
        }
    }
    if (slices <= 1) {
        g.split_stride = 0;
        return bn == 16 ? gemm_launch<16>(g, 1, s) : gemm_launch<128>(g, 1, s);
    }
    // partials at the output's own offsets, one copy per slice
    const long long span = (long long)(g.M - 1) * g.o_m + (long long)(g.N - 1) * g.o_n + 1;
    if ((long long)slices * span > ws_cap) return HGMM_ECAPACITY;
    float* out = g.out_f32;
    g.out_f32 = ws;
    g.split_stride = span;
    const int rc = bn == 16 ? gemm_launch<16>(g, slices, s) : gemm_launch<128>(g, slices, s);
    if (rc) return rc;
    tc::k_sum_slices<<<304, 256, 0, s>>>(ws, slices, span, g.M, g.N, g.n_store, g.o_m, g.o_n, out);
    return cudaGetLastError() == cudaSuccess ? HGMM_OK : HGMM_ECUDA;
}

GemmArgs gargs(const bf16* A, long long a_m, long long a_k, const bf16* B, long long b_n,
               long long b_k, int M, int N, int K, int epi, int* err) {
    GemmArgs g;
    std::memset(&g, 0, sizeof(g));
    g.A = A;
    g.a_m = a_m;
    g.a_k = a_k;
    g.B = B;
    g.b_n = b_n;
    g.b_k = b_k;
    g.M = M;
    g.N = N;
    g.K = K;
    g.n_store = N;
    g.k_split = K;
    g.split_stride = 0;
    g.epi = epi;
    g.err = err;
    return g;
}

// The fused forward (one launch for the three layers; the hidden layers go
// to m->H1 / m->H2 only when the backward pass needs them), or HGMM_ECUDA if
// its tensor maps cannot be encoded (the caller then runs the three GEMMs).
int forward_fused(hgmm_mlp* m, const bf16* X, int batch, float* Y, cudaStream_t s, bool keep_hidden) {
    if (!m->maps) return HGMM_ECUDA;
    CUtensorMap tx, t1, t2, t3, h1 = {}, h2 = {};
    if (!encode_operand(&tx, X, IN, batch, IN, 128) || !encode_operand(&t1, m->W1, IN, HID, IN, HID) ||
        !encode_operand(&t2, m->W2, HID, HID, HID, HID) || !encode_operand(&t3, m->W3, HID, OUTP, HID, OUTP) ||
        (keep_hidden && (!encode_operand(&h1, m->H1, HID, batch, HID, 128) ||
                         !encode_operand(&h2, m->H2, HID, batch, HID, 128))))
        return HGMM_ECUDA;
    k_mlp_forward<<<(batch + 127) / 128, FW_THREADS, FW_SMEM, s>>>(tx, t1, t2, t3, h1, h2, m->P + OFF_B1,
                                                                 m->P + OFF_B2, m->b3p, keep_hidden, Y, batch,
                                                                 m->err);
    return cudaGetLastError() == cudaSuccess ? HGMM_OK : HGMM_ECUDA;
}

int forward_impl(hgmm_mlp* m, const bf16* X, int batch, float* Y, cudaStream_t s, bool keep_hidden = true) {
    if (forward_fused(m, X, batch, Y, s, keep_hidden) == HGMM_OK) return HGMM_OK;
    GemmArgs g = gargs(X, IN, 1, m->W1, IN, 1, batch, HID, IN, tc::EPI_BIAS_RELU_BF16, m->err);
    g.bias = m->P + OFF_B1;
    g.out_bf16 = m->H1;
    g.o_m = HID;
    g.o_n = 1;
    if (int rc = gemm(g, s, nullptr, 0, m->maps)) return rc;
    g = gargs(m->H1, HID, 1, m->W2, HID, 1, batch, HID, HID, tc::EPI_BIAS_RELU_BF16, m->err);
    g.bias = m->P + OFF_B2;
    g.out_bf16 = m->H2;
    g.o_m = HID;
    g.o_n = 1;
    if (int rc = gemm(g, s, nullptr, 0, m->maps)) return rc;
    g = gargs(m->H2, HID, 1, m->W3, HID, 1, batch, OUTP, HID, tc::EPI_BIAS_F32, m->err);
    g.bias = m->b3p;
    g.out_f32 = Y;
    g.o_m = OUT;
    g.o_n = 1;
    g.n_store = OUT;
    return gemm(g, s, nullptr, 0, m->maps);
}

// The backward pass without tensor maps: the fused launches' products one by
// one, the weight gradients into the first slice of ws (with their K slices
// behind it).
int backward_gemms(hgmm_mlp* m, const bf16* X, int batch, cudaStream_t s) {
    float* const part = m->ws + WS_STRIDE;
    const long long part_cap = m->ws_cap - WS_STRIDE;
    // d = a b masked by act > 0, as BF16 (batch x HID)
    auto activation = [&](const bf16* a, long long a_m, const bf16* b, int K, const bf16* act, bf16* d) {
        GemmArgs g = gargs(a, a_m, 1, b, 1, HID, batch, HID, K, tc::EPI_MASK_BF16, m->err);
        g.mask = act;
        g.mask_m = HID;
        g.out_bf16 = d;
        g.o_m = HID;
        g.o_n = 1;
        return gemm(g, s, nullptr, 0, false);
    };
    // columns of a (M) times columns of b (N), summed over the batch
    auto weights = [&](const bf16* a, const bf16* b, long long b_k, int N, int64_t off, long long o_m, long long o_n,
                       int n_store) {
        GemmArgs g = gargs(a, 1, HID, b, 1, b_k, HID, N, batch, tc::EPI_F32, m->err);
        g.out_f32 = m->ws + off;
        g.o_m = o_m;
        g.o_n = o_n;
        g.n_store = n_store;
        return gemm(g, s, part, part_cap, false);
    };
    if (int rc = activation(m->dY, DY_STRIDE, m->W3, OUTP, m->H2, m->dZ2)) return rc;
    if (int rc = activation(m->dZ2, HID, m->W2, HID, m->H1, m->dZ1)) return rc;
    if (int rc = weights(m->H2, m->dY, DY_STRIDE, OUTP, OFF_W3, 1, HID, OUT)) return rc;
    if (int rc = weights(m->dZ2, m->H1, HID, HID, OFF_W2, HID, 1, HID)) return rc;
    return weights(m->dZ1, X, IN, IN, OFF_W1, IN, 1, IN);
}

bool set_gemm_smem() {
    return cudaFuncSetAttribute(tc::k_gemm_bf16<128>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                tc::gemm_smem_bytes(128)) == cudaSuccess &&
           cudaFuncSetAttribute(tc::k_gemm_bf16<16>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                tc::gemm_smem_bytes(16)) == cudaSuccess &&
           cudaFuncSetAttribute(tc::k_gemm_tma<128>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                tc::tma_smem_bytes(128)) == cudaSuccess &&
           cudaFuncSetAttribute(tc::k_gemm_tma<16>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                tc::tma_smem_bytes(16)) == cudaSuccess &&
           cudaFuncSetAttribute(k_mlp_forward, cudaFuncAttributeMaxDynamicSharedMemorySize, FW_SMEM) == cudaSuccess &&
           cudaFuncSetAttribute(k_mlp_backward, cudaFuncAttributeMaxDynamicSharedMemorySize, BW_SMEM) == cudaSuccess &&
           cudaFuncSetAttribute(k_mlp_wgrad, cudaFuncAttributeMaxDynamicSharedMemorySize, WG_SMEM) == cudaSuccess;
}

int check_dev(const hgmm_mlp* m) {
    int cur = -1;
    return (cudaGetDevice(&cur) == cudaSuccess && cur == m->device) ? HGMM_OK : HGMM_EINVAL;
}

WeightCopies copies(const hgmm_mlp* m) { return WeightCopies{m->W1, m->W2, m->W3, m->W2T, m->W3T, m->b3p}; }

// Adam's bias corrections of step t.
void adam_scales(int t, float* c1, float* c2) {
    *c1 = float(1.0 / (1.0 - std::pow(0.9, t)));
    *c2 = float(1.0 / (1.0 - std::pow(0.999, t)));
}

// Loss, gradients and (lr not null) the Adam step of one batch.
int gradients_impl(hgmm_mlp* m, const uint16_t* d_x, const float* d_labels, const int32_t* d_index, int32_t batch,
                   int32_t n_rows, float w_t, float* d_loss, const float* lr, void* stream) {
    if (!m || !d_x || !d_labels || batch < 1 || batch > m->max_batch || !a16(d_x) || !(w_t >= 0.f))
        return HGMM_EINVAL;
    if (d_index && n_rows < 1) return HGMM_EINVAL;
    if (int rc = check_dev(m)) return rc;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const bf16* X = reinterpret_cast<const bf16*>(d_x);
    const float* L = d_labels;
    // tensor maps of the backward pass: K-major operands and the dZ tiles
    // (128-row boxes), and the weight gradients' operands (64-row boxes)
    CUtensorMap bdy = {}, bw3 = {}, bw2 = {}, bz2 = {}, bz1 = {}, gz1 = {}, gx = {}, gz2 = {}, gh1 = {}, gh2 = {},
                gdy = {};
    const bf16* Xb = d_index ? m->Xg : X;
    const bool maps =
        m->maps && encode_operand(&bdy, m->dY, DY_STRIDE, batch, DY_STRIDE, 128) &&
        encode_operand(&bw3, m->W3T, DY_STRIDE, HID, DY_STRIDE, HID) &&
        encode_operand(&bw2, m->W2T, HID, HID, HID, HID) && encode_operand(&bz2, m->dZ2, HID, batch, HID, 128) &&
        encode_operand(&bz1, m->dZ1, HID, batch, HID, 128) && encode_operand(&gz1, m->dZ1, HID, batch, HID, 64) &&
        encode_operand(&gx, Xb, IN, batch, IN, 64) && encode_operand(&gz2, m->dZ2, HID, batch, HID, 64) &&
        encode_operand(&gh1, m->H1, HID, batch, HID, 64) && encode_operand(&gh2, m->H2, HID, batch, HID, 64) &&
        encode_operand(&gdy, m->dY, DY_STRIDE, batch, DY_STRIDE, 64);
    if (d_index) {
        k_gather<<<batch, 160, 0, s>>>(X, d_labels, d_index, n_rows, m->Xg, m->Lg, m->err);
        X = m->Xg;
        L = m->Lg;
    }
    if (int rc = forward_impl(m, X, batch, m->Y, s)) return rc;
    k_loss<<<(batch + LOSS_ROWS - 1) / LOSS_ROWS, LOSS_THREADS, 0, s>>>(m->Y, L, batch, w_t, m->dY, m->dYf,
                                                                       m->loss_part, m->loss_cnt,
                                                                       d_loss ? d_loss : m->loss);
    const int nchunks = (batch + COLSUM_ROWS - 1) / COLSUM_ROWS;
    const int slices = maps ? wg_slices(batch) : 1;
    if (maps) {
        k_mlp_backward<<<(batch + 127) / 128, BW_THREADS, BW_SMEM, s>>>(bdy, bw3, bw2, bz2, bz1, m->H1, m->H2, batch,
                                                                       m->err);
        k_mlp_wgrad<<<WG_TILES * slices + nchunks, WG_THREADS, WG_SMEM, s>>>(
            gz1, gx, gz2, gh1, gh2, gdy, batch, slices, wg_chunks(batch), m->dZ1, m->dZ2, m->dYf, m->ws, m->part, m->err);
    } else {
        if (int rc = backward_gemms(m, X, batch, s)) return rc;
        k_colsum<<<nchunks, WG_THREADS, 0, s>>>(m->dZ1, m->dZ2, m->dYf, batch, m->part);
    }
    constexpr int ug = UPDATE_CTAS + UPDATE_BIAS_CTAS;
    if (lr) {
        m->step += 1;
        float c1, c2;
        adam_scales(m->step, &c1, &c2);
        k_grad_update<true><<<ug, UPDATE_THREADS, 0, s>>>(m->ws, slices, m->part, nchunks, m->G, m->P, m->Mo, m->Vo, *lr, c1,
                                               c2, copies(m));
    } else {
        k_grad_update<false><<<ug, UPDATE_THREADS, 0, s>>>(m->ws, slices, m->part, nchunks, m->G, m->P, m->Mo, m->Vo, 0.f, 0.f,
                                                0.f, copies(m));
    }
    return cudaGetLastError() == cudaSuccess ? HGMM_OK : HGMM_ECUDA;
}

}  // namespace

extern "C" {

int hgmm_mlp_create(int32_t max_batch, hgmm_mlp** out) {
    if (!out) return HGMM_EINVAL;
    *out = nullptr;
    if (max_batch < 1 || max_batch > 65536) return HGMM_EINVAL;
    hgmm_mlp* m = new hgmm_mlp();
    if (cudaGetDevice(&m->device) != cudaSuccess) {
        delete m;
        return HGMM_ECUDA;
    }
    m->max_batch = max_batch;
    const size_t B = size_t(max_batch);
    const int nchunks = (max_batch + COLSUM_ROWS - 1) / COLSUM_ROWS;
    bool good = malloc_into(m, &m->P, N_PARAMS) && malloc_into(m, &m->G, N_PARAMS) &&
                malloc_into(m, &m->Mo, N_PARAMS) && malloc_into(m, &m->Vo, N_PARAMS) &&
                malloc_into(m, &m->W1, size_t(HID) * IN) && malloc_into(m, &m->W2, size_t(HID) * HID) &&
                malloc_into(m, &m->W3, size_t(OUTP) * HID) && malloc_into(m, &m->b3p, OUTP) &&
                malloc_into(m, &m->Xg, B * IN) && malloc_into(m, &m->Lg, B * HGMM_LABEL_FLOATS) &&
                malloc_into(m, &m->H1, B * HID) && malloc_into(m, &m->H2, B * HID) &&
                malloc_into(m, &m->Y, B * OUT) && malloc_into(m, &m->dY, B * DY_STRIDE) &&
                malloc_into(m, &m->dYf, B * OUTP) && malloc_into(m, &m->dZ2, B * HID) &&
                malloc_into(m, &m->dZ1, B * HID) && malloc_into(m, &m->part, size_t(nchunks) * 3 * HID) &&
                malloc_into(m, &m->loss, 1) &&
                malloc_into(m, &m->W2T, size_t(HID) * HID) && malloc_into(m, &m->W3T, size_t(HID) * DY_STRIDE) &&
                malloc_into(m, &m->loss_part, (B + LOSS_ROWS - 1) / LOSS_ROWS) && malloc_into(m, &m->loss_cnt, 1) && malloc_into(m, &m->err, 1) &&
                malloc_into(m, &m->prop_x, IN) && malloc_into(m, &m->prop_fr, 2 * HGMM_FRAME_DOUBLES) &&
                malloc_into(m, &m->prop_y, 16);
    // the fused launch's slices, or without tensor maps the gradients and dW1's 16 slices
    m->ws_cap = std::max<long long>(WG_MAX_SLICES * WS_STRIDE, WS_STRIDE + 16ll * HID * IN);
    good = good && malloc_into(m, &m->ws, size_t(m->ws_cap));
    good = good && set_gemm_smem();
    if (!good) {
        hgmm_mlp_destroy(m);
        return HGMM_ENOMEM;
    }
    *out = m;
    return HGMM_OK;
}

void hgmm_mlp_destroy(hgmm_mlp* m) {
    if (!m) return;
    int cur = 0;
    cudaGetDevice(&cur);
    cudaSetDevice(m->device);
    for (void* p : m->allocs) cudaFree(p);
    cudaSetDevice(cur);
    delete m;
}

int hgmm_mlp_set_params(hgmm_mlp* m, const float* h_params, int64_t count) {
    if (!m || !h_params || count != N_PARAMS) return HGMM_EINVAL;
    if (int rc = check_dev(m)) return rc;
    const size_t bytes = size_t(N_PARAMS) * sizeof(float);
    bool good = cudaMemcpy(m->P, h_params, bytes, cudaMemcpyHostToDevice) == cudaSuccess &&
                cudaMemset(m->Mo, 0, bytes) == cudaSuccess && cudaMemset(m->Vo, 0, bytes) == cudaSuccess &&
                cudaMemset(m->G, 0, bytes) == cudaSuccess;
    if (!good) return HGMM_ECUDA;
    k_refresh<<<512, 256>>>(m->P, copies(m));
    m->step = 0;
    return cudaDeviceSynchronize() == cudaSuccess ? HGMM_OK : HGMM_ECUDA;
}

int hgmm_mlp_get_params(hgmm_mlp* m, float* h_params, int64_t count) {
    if (!m || !h_params || count != N_PARAMS) return HGMM_EINVAL;
    if (cudaDeviceSynchronize() != cudaSuccess) return HGMM_ECUDA;
    return cudaMemcpy(h_params, m->P, size_t(N_PARAMS) * sizeof(float), cudaMemcpyDeviceToHost) == cudaSuccess
               ? HGMM_OK
               : HGMM_ECUDA;
}

int hgmm_mlp_read_grads(hgmm_mlp* m, float* h_grads, int64_t count) {
    if (!m || !h_grads || count != N_PARAMS) return HGMM_EINVAL;
    if (cudaDeviceSynchronize() != cudaSuccess) return HGMM_ECUDA;
    return cudaMemcpy(h_grads, m->G, size_t(N_PARAMS) * sizeof(float), cudaMemcpyDeviceToHost) == cudaSuccess
               ? HGMM_OK
               : HGMM_ECUDA;
}

int hgmm_mlp_forward(hgmm_mlp* m, const uint16_t* d_x, int32_t batch, float* d_y, void* stream) {
    if (!m || !d_x || !d_y || batch < 1 || batch > m->max_batch || !a16(d_x)) return HGMM_EINVAL;
    if (int rc = check_dev(m)) return rc;
    return forward_impl(m, reinterpret_cast<const bf16*>(d_x), batch, d_y, static_cast<cudaStream_t>(stream),
                        false);
}

int hgmm_mlp_gradients(hgmm_mlp* m, const uint16_t* d_x, const float* d_labels, const int32_t* d_index,
                       int32_t batch, int32_t n_rows, float w_t, float* d_loss, void* stream) {
    return gradients_impl(m, d_x, d_labels, d_index, batch, n_rows, w_t, d_loss, nullptr, stream);
}

int hgmm_mlp_adam(hgmm_mlp* m, float lr, void* stream) {
    if (!m || !(lr >= 0.f)) return HGMM_EINVAL;
    if (int rc = check_dev(m)) return rc;
    m->step += 1;
    float c1, c2;
    adam_scales(m->step, &c1, &c2);
    k_adam<<<608, 256, 0, static_cast<cudaStream_t>(stream)>>>(m->P, m->G, m->Mo, m->Vo, lr, c1, c2, copies(m));
    return cudaGetLastError() == cudaSuccess ? HGMM_OK : HGMM_ECUDA;
}

int hgmm_mlp_train_step(hgmm_mlp* m, const uint16_t* d_x, const float* d_labels, const int32_t* d_index,
                        int32_t batch, int32_t n_rows, float w_t, float lr, float* d_loss, void* stream) {
    if (!(lr >= 0.f)) return HGMM_EINVAL;
    return gradients_impl(m, d_x, d_labels, d_index, batch, n_rows, w_t, d_loss, &lr, stream);
}

int hgmm_mlp_sync(hgmm_mlp* m, void* stream) {
    if (!m) return HGMM_EINVAL;
    if (cudaStreamSynchronize(static_cast<cudaStream_t>(stream)) != cudaSuccess) return HGMM_ECUDA;
    int e = 0;
    if (cudaMemcpy(&e, m->err, sizeof(int), cudaMemcpyDeviceToHost) != cudaSuccess ||
        cudaMemset(m->err, 0, sizeof(int)) != cudaSuccess)
        return HGMM_ECUDA;
    if (e & ERR_TIMEOUT) return HGMM_ETIMEOUT;
    if (e & ERR_INDEX) return HGMM_EINVAL;
    return HGMM_OK;
}

int hgmm_tree_features(hgmm_tree* t, uint16_t* d_feat, double* d_frame, void* stream) {
    if (!t || !d_feat || !d_frame || !t->built || t->depth < 2 || !a16(d_feat)) return HGMM_EINVAL;
    const FeatJob j{t->root, t->stat, reinterpret_cast<bf16*>(d_feat), d_frame};
    k_tree_features<<<1, FEAT_NODES, 0, static_cast<cudaStream_t>(stream)>>>(j, j);
    return cudaGetLastError() == cudaSuccess ? HGMM_OK : HGMM_ECUDA;
}

int hgmm_propose(hgmm_tree* tgt, hgmm_tree* src, hgmm_mlp* m, void* stream, double* d_T_out) {
    if (!tgt || !src || !m || !d_T_out) return HGMM_EINVAL;
    if (int rc = check_dev(m)) return rc;
    if (!src->built || src->depth < 2 || !tgt->built || tgt->depth < 2) return HGMM_EINVAL;
    // network input: [features(source), features(target)], frames likewise,
    // both trees in one launch
    k_tree_features<<<2, FEAT_NODES, 0, static_cast<cudaStream_t>(stream)>>>(
        FeatJob{src->root, src->stat, m->prop_x, m->prop_fr},
        FeatJob{tgt->root, tgt->stat, m->prop_x + FEAT_PER_CLOUD, m->prop_fr + FRAME_DOUBLES});
    if (cudaGetLastError() != cudaSuccess) return HGMM_ECUDA;
    if (int rc = hgmm_mlp_forward(m, reinterpret_cast<const uint16_t*>(m->prop_x), 1, m->prop_y, stream)) return rc;
    return hgmm_pose_decode(m->prop_y, m->prop_fr, 1, d_T_out, stream);
}

int hgmm_pose_decode(const float* d_y, const double* d_frames, int32_t n, double* d_T, void* stream) {
    if (!d_y || !d_frames || !d_T || n < 1) return HGMM_EINVAL;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (n <= DECODE_FEW)
        k_decode<<<(n + DECODE_THREADS / 16 - 1) / (DECODE_THREADS / 16), DECODE_THREADS, 0, s>>>(d_y, d_frames, n,
                                                                                                  d_T);
    else
        k_decode_many<<<(n + DECODE_THREADS - 1) / DECODE_THREADS, DECODE_THREADS, 0, s>>>(d_y, d_frames, n, d_T);
    return cudaGetLastError() == cudaSuccess ? HGMM_OK : HGMM_ECUDA;
}

int hgmm_pose_encode(const double* d_T, const double* d_frames, int32_t n, float* d_labels, void* stream) {
    if (!d_T || !d_frames || !d_labels || n < 1) return HGMM_EINVAL;
    k_encode<<<(n + 127) / 128, 128, 0, static_cast<cudaStream_t>(stream)>>>(d_T, d_frames, n, d_labels);
    return cudaGetLastError() == cudaSuccess ? HGMM_OK : HGMM_ECUDA;
}

int hgmm_debug_mlp_maps(hgmm_mlp* m, int32_t enable) {
    if (!m) return HGMM_EINVAL;
    m->maps = enable != 0;
    return HGMM_OK;
}

int hgmm_debug_gemm(const uint16_t* d_A, int64_t a_m, int64_t a_k, const uint16_t* d_B, int64_t b_n,
                    int64_t b_k, int32_t M, int32_t N, int32_t K, float* d_out, void* stream) {
    if (!d_A || !d_B || !d_out) return HGMM_EINVAL;
    static int* err = nullptr;  // error word of the checking launches
    if (!err && (cudaMalloc(&err, sizeof(int)) != cudaSuccess || cudaMemset(err, 0, sizeof(int)) != cudaSuccess))
        return HGMM_ECUDA;
    static bool attr = false;
    static float* ws = nullptr;
    const long long ws_cap = (long long)MAX_SLICES * 256 * 1536;
    if (!attr) {
        if (!set_gemm_smem() || cudaMalloc(&ws, size_t(ws_cap) * sizeof(float)) != cudaSuccess) return HGMM_ECUDA;
        attr = true;
    }
    GemmArgs g = gargs(reinterpret_cast<const bf16*>(d_A), a_m, a_k, reinterpret_cast<const bf16*>(d_B),
                       b_n, b_k, M, N, K, tc::EPI_F32, err);
    g.out_f32 = d_out;
    g.o_m = N;
    g.o_n = 1;
    return gemm(g, static_cast<cudaStream_t>(stream), ws, ws_cap);
}

int hgmm_pose_select(int32_t n, const double* d_T_a, const double* d_obj_a, const double* d_T_b,
                     const double* d_obj_b, double* d_T_out, int32_t* d_choice, double* d_obj_out,
                     void* stream) {
    if (n < 1 || !d_T_a || !d_obj_a || !d_T_b || !d_obj_b || !d_T_out) return HGMM_EINVAL;
    k_select<<<(n + 127) / 128, 128, 0, static_cast<cudaStream_t>(stream)>>>(n, d_T_a, d_obj_a, d_T_b,
                                                                             d_obj_b, d_T_out, d_choice,
                                                                             d_obj_out);
    return cudaGetLastError() == cudaSuccess ? HGMM_OK : HGMM_ECUDA;
}

int hgmm_pose_compose(int32_t n, const double* d_A, const double* d_B, double* d_out, void* stream) {
    if (n < 1 || !d_A || !d_B || !d_out || d_out == d_A || d_out == d_B) return HGMM_EINVAL;
    k_compose<<<(n + 127) / 128, 128, 0, static_cast<cudaStream_t>(stream)>>>(n, d_A, d_B, d_out);
    return cudaGetLastError() == cudaSuccess ? HGMM_OK : HGMM_ECUDA;
}

}  // extern "C"
