// Backward pass of the pose-proposal network on the tensor cores, included by
// hgmm_mlp.cu after its constants and parameter offsets.
//
// A training step is latency: 1024 rows are 2.4 GFLOP (1.3 us at the measured
// BF16 rate) and a few MB.  Its parts are therefore few launches that each
// fill the chip: the loss (four lanes per row), one launch for both
// activation gradients of a 128-row block, one for all weight and bias
// gradients, one that sums the K slices and applies Adam.  A step of 1,024
// rows takes 57 us; with one GEMM launch per product, the loss in one CTA and
// separate column sums and slice sums it took 246.  Of the 57, alone and with
// cold caches: forward 19, loss 9, backward 15, weight gradients 9, update 8.
#pragma once

namespace hgmm {
namespace {

constexpr int DY_STRIDE = 64;      // BF16 row of dY: nine values, then zeros (one 128-byte swizzled row)
constexpr int LOSS_THREADS = 128;  // 32 rows per CTA
constexpr int LOSS_ROWS = LOSS_THREADS / 4;

// Sum over the lanes of a quad.
__device__ __forceinline__ double quad_sum(double v) {
    v += __shfl_xor_sync(0xffffffffu, v, 1);
    return v + __shfl_xor_sync(0xffffffffu, v, 2);
}

// Loss of every row and dL/dy (mean over the batch), four lanes per row: lane
// i < 3 holds component i of every vector, so a vector operation is one FP64
// warp instruction for eight rows (an FP64 warp instruction holds its pipe for
// about 64 cycles whatever its active lanes: one thread per row in one CTA
// took 64 us for 1024 rows).  The row losses are summed in a fixed order: in
// the CTA, then over the CTAs by the last one to finish.
__global__ void __launch_bounds__(LOSS_THREADS)
k_loss(const float* __restrict__ Y, const float* __restrict__ L, int batch, float w_t, bf16* __restrict__ dY,
       float* __restrict__ dYf, double* __restrict__ part, unsigned* __restrict__ cnt, float* __restrict__ loss) {
    __shared__ double red[LOSS_THREADS];
    __shared__ bool last;
    const int lane = threadIdx.x & 31, i = lane & 3, q0 = lane & ~3;
    const int r = blockIdx.x * LOSS_ROWS + (threadIdx.x >> 2);
    const bool own = r < batch && i < 3;
    const double inv_b = 1.0 / double(batch);
    double a1 = 0.0, a2 = 0.0, yt = 0.0, l0 = 0.0, l1 = 0.0, l2 = 0.0, lt = 0.0;
    if (own) {
        const float* y = Y + int64_t(r) * OUT;
        const float* l = L + int64_t(r) * HGMM_LABEL_FLOATS;
        a1 = y[i];
        a2 = y[3 + i];
        yt = y[6 + i];
        // label R' row-major: column k entry i at l[3 i + k]
        l0 = l[3 * i];
        l1 = l[3 * i + 1];
        l2 = l[3 * i + 2];
        lt = l[9 + i];
    }
    const int nx = i < 3 ? q0 + (i == 2 ? 0 : i + 1) : lane, pv = i < 3 ? q0 + (i == 0 ? 2 : i - 1) : lane;
    auto cross = [&](double x, double y) {
        const double xn = __shfl_sync(0xffffffffu, x, nx), xp = __shfl_sync(0xffffffffu, x, pv);
        const double yn = __shfl_sync(0xffffffffu, y, nx), yp = __shfl_sync(0xffffffffu, y, pv);
        return xn * yp - xp * yn;
    };
    // Gram-Schmidt of (a1, a2) into b1, b2, b3 = b1 x b2
    const double s1 = quad_sum(a1 * a1);
    const double i1 = s1 > 0.0 ? rsqrt_f64(s1) : 0.0;
    const double b1 = a1 * i1;
    const double dd = quad_sum(b1 * a2);
    const double u = a2 - dd * b1;
    const double s2 = quad_sum(u * u);
    const double i2 = s2 > 0.0 ? rsqrt_f64(s2) : 0.0;
    const double b2 = u * i2;
    const double b3 = cross(b1, b2);
    const double r0 = b1 - l0, r1 = b2 - l1, r2 = b3 - l2, d = yt - lt;
    const double e = own ? r0 * r0 + r1 * r1 + r2 * r2 + double(w_t) * d * d : 0.0;
    const double G1 = 2.0 * r0, G2 = 2.0 * r1, G3 = 2.0 * r2, gt = 2.0 * double(w_t) * d;
    // back through b3 = b1 x b2, b2 = u / |u|, u = a2 - (b1.a2) b1, b1 = a1 / |a1|
    double gb1 = G1 + cross(b2, G3);
    const double gb2 = G2 + cross(G3, b1);
    const double gu = (gb2 - quad_sum(gb2 * b2) * b2) * i2;
    const double q = quad_sum(gu * b1);
    const double ga2 = gu - q * b1;
    gb1 += -q * a2 - dd * gu;
    const double p1 = quad_sum(gb1 * b1);
    if (own) {
        const double g[3] = {(gb1 - p1 * b1) * i1 * inv_b, ga2 * inv_b, gt * inv_b};
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            dYf[int64_t(r) * OUTP + 3 * k + i] = float(g[k]);
            dY[int64_t(r) * DY_STRIDE + 3 * k + i] = __double2bfloat16(g[k]);
        }
    }
    red[threadIdx.x] = e;
    __syncthreads();
    if (threadIdx.x < 32) {
        double s = red[lane];
#pragma unroll
        for (int k = 1; k < LOSS_THREADS / 32; ++k) s += red[lane + 32 * k];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (lane == 0) {
            part[blockIdx.x] = s;
            __threadfence();
            last = atomicAdd(cnt, 1u) == gridDim.x - 1;
        }
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    double s = 0.0;
    for (int b = threadIdx.x; b < int(gridDim.x); b += LOSS_THREADS) s += __ldcg(part + b);
    red[threadIdx.x] = s;
    __syncthreads();
    if (threadIdx.x < 32) {
        s = red[lane];
#pragma unroll
        for (int k = 1; k < LOSS_THREADS / 32; ++k) s += red[lane + 32 * k];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (lane == 0) {
            if (loss) *loss = float(s * inv_b);
            *cnt = 0u;  // ready for the next launch
        }
    }
}

// --------------------------------------------------- bulk stores and MN-major operands
__device__ __forceinline__ void bulk_s2g(void* dst, uint32_t src, uint32_t bytes) {
    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" :: "l"(dst), "r"(src), "r"(bytes)
                 : "memory");
}
// Descriptor of an operand stored with M (or N) contiguous, in the 128-byte
// swizzled layout of a TMA box of 64 columns: K rows of 128 bytes, groups of
// eight rows 1024 bytes apart (stride byte offset), the next 64 columns one
// box further (leading byte offset).  The instruction descriptor's transpose
// bits (15: A, 16: B) select this layout.
__device__ __forceinline__ uint64_t smem_desc_mn(uint32_t addr, uint32_t box_bytes) {
    return uint64_t((addr >> 4) & 0x3FFFu) | (uint64_t((box_bytes >> 4) & 0x3FFFu) << 16) |
           (uint64_t(1024 >> 4) << 32) | (uint64_t(1) << 46) | (uint64_t(2) << 61);
}

// ------------------------------------------------------- activation gradients
// dZ2 = (dY W3) * [H2 > 0] and dZ1 = (dZ2 W2) * [H1 > 0] of one 128-row block:
// dY, W3^T and three of the four W2^T tiles are loaded up front (the fourth
// takes W3^T's place), the first product is a single K = 16 step, and dZ2
// reaches the second one through shared memory in the swizzled layout that
// TMA also stores it to global memory from.  Eight epilogue warps: warp w
// owns TMEM lanes 32 (w mod 4).. and the columns' half w / 4.
constexpr int BW_THREADS = 320;
constexpr int BW_DY = FW_H;
constexpr int BW_W3 = BW_DY + FW_A;
constexpr int BW_W2 = BW_W3 + FW_B;
constexpr int BW_SMEM = BW_W2 + 3 * FW_B + 1024;

__device__ __forceinline__ void bw_epilogue(uint32_t tacc, const bf16* __restrict__ act, uint32_t zbuf, int r,
                                            int half) {
#pragma unroll 1
    for (int c = 2 * half; c < 2 * half + 2; ++c) {
        float v[64];
        tc::tmem_ld64(tacc + uint32_t(c * 64), v);
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const uint4 a = act ? __ldg(reinterpret_cast<const uint4*>(act + c * 64) + u) : make_uint4(0u, 0u, 0u, 0u);
            const uint32_t aw[4] = {a.x, a.y, a.z, a.w};
            uint32_t w[4];
#pragma unroll
            for (int h = 0; h < 4; ++h) {
                const float lo = __uint_as_float(aw[h] << 16), hi = __uint_as_float(aw[h] & 0xffff0000u);
                const __nv_bfloat162 p = __floats2bfloat162_rn(lo > 0.f ? v[8 * u + 2 * h] : 0.f,
                                                               hi > 0.f ? v[8 * u + 2 * h + 1] : 0.f);
                w[h] = *reinterpret_cast<const uint32_t*>(&p);
            }
            asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};"
                         :: "r"(zbuf + uint32_t(c * FW_A) + sw128_offset(r, u)), "r"(w[0]), "r"(w[1]), "r"(w[2]),
                            "r"(w[3]) : "memory");
        }
    }
}

__global__ void __launch_bounds__(BW_THREADS, 1)
k_mlp_backward(const __grid_constant__ CUtensorMap tmDY, const __grid_constant__ CUtensorMap tmW3T,
               const __grid_constant__ CUtensorMap tmW2T, const __grid_constant__ CUtensorMap tmZ2,
               const __grid_constant__ CUtensorMap tmZ1, const bf16* __restrict__ H1, const bf16* __restrict__ H2,
               int batch, int* __restrict__ err) {
    extern __shared__ unsigned char bw_raw[];
    __shared__ __align__(8) uint64_t full1, full2[4], done1, done2, z_ready;
    __shared__ uint32_t tmem_slot;
    __shared__ int fail;
    const uint32_t base = (tc::smem_u32(bw_raw) + 1023u) & ~1023u;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int m0 = blockIdx.x * 128;
    constexpr int NK2 = HID / 64;
    constexpr uint32_t ID = tc::idesc_bf16_f32(128, HID);
    if (warp == 8) {
        tc::tmem_alloc(&tmem_slot, 512);
        tc::tmem_relinquish();
    }
    if (threadIdx.x == 288) {
        tc::mbar_init(&full1, 1);
        for (int i = 0; i < 4; ++i) tc::mbar_init(&full2[i], 1);
        tc::mbar_init(&done1, 1);
        tc::mbar_init(&done2, 1);
        tc::mbar_init(&z_ready, 256);
        fail = 0;
        tc::fence_mbar_init();
        tc::prefetch_tmap(&tmDY);
        tc::prefetch_tmap(&tmW3T);
        tc::prefetch_tmap(&tmW2T);
        tc::prefetch_tmap(&tmZ2);
        tc::prefetch_tmap(&tmZ1);
    }
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t tmem = tmem_slot;
    auto w2_tile = [&](int kt) { return base + (kt < 3 ? BW_W2 + kt * FW_B : BW_W3); };
    int issued2 = 0;
    if (threadIdx.x == 256) {
        tc::mbar_arrive_expect_tx(&full1, uint32_t(FW_A + FW_B));
        tc::tma_load_2d(base + BW_DY, &tmDY, 0, m0, &full1);
        tc::tma_load_2d(base + BW_W3, &tmW3T, 0, 0, &full1);
        for (int kt = 0; kt < NK2; ++kt) {
            if (kt == 3 && !fw_wait(&done1, 0, &fail)) break;  // the last tile goes where W3^T was
            tc::mbar_arrive_expect_tx(&full2[kt], uint32_t(FW_B));
            tc::tma_load_2d(w2_tile(kt), &tmW2T, kt * 64, 0, &full2[kt]);
            issued2 = kt + 1;
        }
    } else if (warp == 9) {
        const bool lead = tc::elect_one();
        bool ok = __all_sync(0xffffffffu, fw_wait(&full1, 0, &fail));
        if (lead) {
            if (ok) {
                tc::fence_after_sync();
                tc::mma_bf16(tmem, tc::smem_desc_sw128(base + BW_DY), tc::smem_desc_sw128(base + BW_W3), ID, 0u);
            }
            tc::mma_commit(&done1);
        }
        __syncwarp();
        ok = ok && __all_sync(0xffffffffu, fw_wait(&z_ready, 0, &fail));
        for (int kt = 0; kt < NK2 && ok; ++kt) {
            ok = __all_sync(0xffffffffu, fw_wait(&full2[kt], 0, &fail));
            if (!ok) break;
            tc::fence_after_sync();
            mma_k64(lead, tmem + 256u, tc::smem_desc_sw128(base + kt * FW_A), tc::smem_desc_sw128(w2_tile(kt)), ID,
                    kt != 0, nullptr);
        }
        if (lead) tc::mma_commit(&done2);
    } else if (warp < 8) {
        const int r = (warp & 3) * 32 + lane, half = warp >> 2, m = m0 + r;
        const uint32_t lanes = uint32_t((warp & 3) * 32) << 16;
        const bool row = m < batch;
        const bool ok1 = __all_sync(0xffffffffu, fw_wait(&done1, 0, &fail));
        if (ok1) {
            tc::fence_after_sync();
            bw_epilogue(tmem + lanes, row ? H2 + int64_t(m) * HID : nullptr, base, r, half);
            tc::fence_before_sync();
        }
        tc::fence_proxy_async();  // dZ2, written here, is read by the tensor core and by TMA
        asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" :: "r"(tc::smem_u32(&z_ready)) : "memory");
        asm volatile("bar.sync 1, 256;" ::: "memory");
        if (threadIdx.x == 0 && ok1) {
            for (int c = 0; c < 4; ++c) tma_store_2d(&tmZ2, c * 64, m0, base + c * FW_A);
            bulk_commit();
        }
        const bool ok2 = __all_sync(0xffffffffu, ok1 && fw_wait(&done2, 0, &fail));
        if (threadIdx.x == 0) bulk_wait_read();  // dZ2 has left the buffer that dZ1 now takes
        asm volatile("bar.sync 1, 256;" ::: "memory");
        if (ok2) {
            tc::fence_after_sync();
            bw_epilogue(tmem + lanes + 256u, row ? H1 + int64_t(m) * HID : nullptr, base, r, half);
            tc::fence_before_sync();
        }
        tc::fence_proxy_async();
        asm volatile("bar.sync 1, 256;" ::: "memory");
        if (threadIdx.x == 0) {
            if (ok2) {
                for (int c = 0; c < 4; ++c) tma_store_2d(&tmZ1, c * 64, m0, base + c * FW_A);
                bulk_commit();
            }
            bulk_wait();
        }
    }
    __syncwarp();
    if (threadIdx.x == 256) {  // loads issued but perhaps not consumed: let them land
        tc::mbar_wait_bounded(&full1, 0, tc::MBAR_SPIN_LIMIT);
        for (int kt = 0; kt < issued2; ++kt) tc::mbar_wait_bounded(&full2[kt], 0, tc::MBAR_SPIN_LIMIT);
    }
    if (threadIdx.x == 288) tc::mbar_wait_bounded(&done2, 0, tc::MBAR_SPIN_LIMIT);
    __syncthreads();
    if (threadIdx.x == 0 && *(volatile int*)&fail) atomicOr(err, ERR_TIMEOUT);
    tc::fence_before_sync();
    __syncthreads();
    if (warp == 8) tc::tmem_dealloc(tmem, 512);
}

// ----------------------------------------------------------- weight gradients
// dW1 = dZ1^T X, dW2 = dZ2^T H1 and dW3^T = H2^T dY in one launch, K (the
// batch) cut into slices, and the bias gradients' partial column sums on
// further CTAs.  Every operand is read where it lies, with M or N contiguous,
// by TMA boxes of 64 columns x 64 rows; rows past the batch read zero.  A CTA
// owns a tile of one slice (128 x 256 of dW1, 128 x 128 of dW2, 128 x 64 of
// dW3) and writes it to its slice's partials with one bulk copy per row, staged
// through the operand ring (rows 1040 bytes apart: no bank conflicts).
//
// The tensor core rounds its FP32 sums towards zero at every step, so a sum's
// error grows with the number of rows that one accumulator takes.  A slice is
// therefore cut once more, into as many accumulators as TMEM's 512 columns
// hold (two for dW1, four for dW2 and dW3), added in FP32 when the tile is
// read back: at most 1/16 (dW1) or 1/32 of the batch per accumulator.  Error of
// dW1 / dW2 / dW3 against float64 on operands that BF16 holds exactly, 4,096
// rows: 2.0e-7 / 1.0e-7 / 1.2e-7, with one accumulator per slice 4.6e-7 / 4.4e-7 /
// 5.2e-7 (and 1 us less for a step of 1,024 to 4,096 rows: 57.3 against 58.4).
constexpr int WG_THREADS = 256;
constexpr int WG_STAGES = 4;
constexpr int WG_BOX = 64 * 128;             // 64 rows x 64 BF16
constexpr int WG_STAGE = 6 * WG_BOX;         // two A boxes, up to four B boxes
constexpr int WG_ROW = 1040;
constexpr int WG_SMEM = WG_STAGES * WG_STAGE + 1024;
static_assert(OFF_B1 % 4 == 0 && OFF_W2 % 4 == 0 && OFF_B2 % 4 == 0 && OFF_W3 % 4 == 0 && OFF_B3 % 4 == 0,
              "whole vectors of weights");
static_assert(128 * WG_ROW <= WG_STAGES * WG_STAGE, "staging inside the ring");
constexpr int WG_TILES1 = 2 * (IN / 256), WG_TILES2 = 2 * (HID / 128);
constexpr int WG_TILES = WG_TILES1 + WG_TILES2 + 2;
constexpr int WG_MAX_SLICES = 8;
constexpr int WG_ACC1 = 2, WG_ACC23 = 4;     // accumulators per CTA of dW1; of dW2 and dW3
static_assert(WG_ACC1 * 256 <= 512 && WG_ACC23 * 128 <= 512, "TMEM columns");
constexpr int64_t WS_STRIDE = (N_PARAMS + 3) / 4 * 4;

// K slices of a batch: 64-row chunks per slice (the tiles times the slices
// are at most 128 CTAs: one wave beside the column sums).
inline int wg_chunks(int batch) { return ((batch + 63) / 64 + WG_MAX_SLICES - 1) / WG_MAX_SLICES; }
inline int wg_slices(int batch) {
    const int c = wg_chunks(batch);
    return ((batch + 63) / 64 + c - 1) / c;
}

__device__ __forceinline__ void colsum_chunk(const bf16* __restrict__ dZ1, const bf16* __restrict__ dZ2,
                                             const float* __restrict__ dYf, int batch, int chunk,
                                             float* __restrict__ part) {
    const int j = threadIdx.x, r0 = chunk * COLSUM_ROWS, r1 = min(batch, r0 + COLSUM_ROWS);
    float s1 = 0.f, s2 = 0.f, sy = 0.f;
#pragma unroll 16
    for (int r = r0; r < r1; ++r) {
        s1 += __bfloat162float(dZ1[int64_t(r) * HID + j]);
        s2 += __bfloat162float(dZ2[int64_t(r) * HID + j]);
    }
    if (j < OUTP)
        for (int r = r0; r < r1; ++r) sy += dYf[int64_t(r) * OUTP + j];
    float* p = part + int64_t(chunk) * 3 * HID + j;
    p[0] = s1;
    p[HID] = s2;
    p[2 * HID] = sy;
}

// The column sums alone (without tensor maps).
__global__ void __launch_bounds__(WG_THREADS)
k_colsum(const bf16* __restrict__ dZ1, const bf16* __restrict__ dZ2, const float* __restrict__ dYf, int batch,
         float* __restrict__ part) {
    colsum_chunk(dZ1, dZ2, dYf, batch, int(blockIdx.x), part);
}

__global__ void __launch_bounds__(WG_THREADS, 1)
k_mlp_wgrad(const __grid_constant__ CUtensorMap tmZ1, const __grid_constant__ CUtensorMap tmX,
            const __grid_constant__ CUtensorMap tmZ2, const __grid_constant__ CUtensorMap tmH1,
            const __grid_constant__ CUtensorMap tmH2, const __grid_constant__ CUtensorMap tmDY, int batch, int slices,
            int chunks, const bf16* __restrict__ dZ1, const bf16* __restrict__ dZ2, const float* __restrict__ dYf,
            float* __restrict__ ws, float* __restrict__ part, int* __restrict__ err) {
    extern __shared__ unsigned char wg_raw[];
    __shared__ __align__(8) uint64_t full[WG_STAGES], empty[WG_STAGES], done;
    __shared__ uint32_t tmem_slot;
    __shared__ int fail;
    const int gemm_ctas = WG_TILES * slices;
    if (int(blockIdx.x) >= gemm_ctas) {
        colsum_chunk(dZ1, dZ2, dYf, batch, int(blockIdx.x) - gemm_ctas, part);
        return;
    }
    const uint32_t base = (tc::smem_u32(wg_raw) + 1023u) & ~1023u;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int tile = blockIdx.x / slices, slice = blockIdx.x % slices;
    // tile -> product, first column of A (rows of D) and of B (columns of D), columns
    const int which = tile < WG_TILES1 ? 0 : (tile < WG_TILES1 + WG_TILES2 ? 1 : 2);
    const int m0 = 128 * (tile & 1);
    const int n0 = which == 0 ? 256 * (tile >> 1) : (which == 1 ? 128 * ((tile - WG_TILES1) >> 1) : 0);
    const int width = which == 0 ? 256 : (which == 1 ? 128 : 64);
    const int nb = width / 64;
    const void* ta = which == 0 ? &tmZ1 : (which == 1 ? &tmZ2 : &tmH2);
    const void* tb = which == 0 ? &tmX : (which == 1 ? &tmH1 : &tmDY);
    const uint32_t idesc = tc::idesc_bf16_f32(128, width) | (1u << 15) | (1u << 16);
    const int k0 = slice * chunks, nk = min(chunks, (batch + 63) / 64 - k0);
    // chunks per accumulator, and accumulators in use
    const int per_acc = (chunks + (which == 0 ? WG_ACC1 : WG_ACC23) - 1) / (which == 0 ? WG_ACC1 : WG_ACC23);
    const int accs = (nk + per_acc - 1) / per_acc;
    if (warp == 4) {
        tc::tmem_alloc(&tmem_slot, 512);
        tc::tmem_relinquish();
    }
    if (threadIdx.x == 160) {
        for (int i = 0; i < WG_STAGES; ++i) {
            tc::mbar_init(&full[i], 1);
            tc::mbar_init(&empty[i], 1);
        }
        tc::mbar_init(&done, 1);
        fail = 0;
        tc::fence_mbar_init();
        tc::prefetch_tmap(ta);
        tc::prefetch_tmap(tb);
    }
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t tmem = tmem_slot;
    int issued = 0;
    if (threadIdx.x == 128) {
        for (int kt = 0; kt < nk; ++kt) {
            const int st = kt % WG_STAGES;
            if (kt >= WG_STAGES && !fw_wait(&empty[st], ((kt / WG_STAGES) - 1) & 1, &fail)) break;
            const uint32_t sa = base + st * WG_STAGE;
            const int row = (k0 + kt) * 64;
            tc::mbar_arrive_expect_tx(&full[st], uint32_t((2 + nb) * WG_BOX));
            for (int b = 0; b < 2; ++b) tc::tma_load_2d(sa + b * WG_BOX, ta, m0 + 64 * b, row, &full[st]);
            for (int b = 0; b < nb; ++b) tc::tma_load_2d(sa + (2 + b) * WG_BOX, tb, n0 + 64 * b, row, &full[st]);
            issued = kt + 1;
        }
    } else if (warp == 5) {
        const bool lead = tc::elect_one();
        for (int kt = 0; kt < nk; ++kt) {
            const int st = kt % WG_STAGES;
            if (!__all_sync(0xffffffffu, fw_wait(&full[st], (kt / WG_STAGES) & 1, &fail))) break;
            tc::fence_after_sync();
            const uint32_t sa = base + st * WG_STAGE;
            const uint64_t da = smem_desc_mn(sa, WG_BOX), db = smem_desc_mn(sa + 2 * WG_BOX, WG_BOX);
            const int acc = kt / per_acc;
            const bool first = kt == acc * per_acc;
            if (lead) {
#pragma unroll
                for (int kk = 0; kk < 4; ++kk)  // 16 rows of 128 bytes
                    tc::mma_bf16(tmem + uint32_t(acc * width), da + 128 * kk, db + 128 * kk, idesc,
                                 !first || kk != 0 ? 1u : 0u);
                tc::mma_commit(&empty[st]);
            }
            __syncwarp();
        }
        if (lead) tc::mma_commit(&done);
    } else if (warp < 4) {
        const int r = warp * 32 + lane, m = m0 + r;
        const uint32_t tacc = tmem + (uint32_t(warp * 32) << 16);
        float* out = ws + slice * WS_STRIDE;
        // after `done` nothing reads the ring any more: every load was consumed
        if (__all_sync(0xffffffffu, fw_wait(&done, 0, &fail) && !*(volatile int*)&fail)) {
            tc::fence_after_sync();
            if (which == 2) {
                float v[16];
                tc::tmem_ld16(tacc, v);
                for (int q = 1; q < accs; ++q) {
                    float x[16];
                    tc::tmem_ld16(tacc + uint32_t(q * width), x);
#pragma unroll
                    for (int o = 0; o < OUT; ++o) v[o] += x[o];
                }
#pragma unroll
                for (int o = 0; o < OUT; ++o) out[OFF_W3 + o * HID + m] = v[o];
            } else {
                const uint32_t row = base + uint32_t(r * WG_ROW);
#pragma unroll 1
                for (int c = 0; c < nb; ++c) {
                    float v[64];
                    tc::tmem_ld64(tacc + uint32_t(64 * c), v);
#pragma unroll 1
                    for (int q = 1; q < accs; ++q) {
                        float x[64];
                        tc::tmem_ld64(tacc + uint32_t(q * width + 64 * c), x);
#pragma unroll
                        for (int o = 0; o < 64; ++o) v[o] += x[o];
                    }
#pragma unroll
                    for (int q = 0; q < 16; ++q)
                        asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};"
                                     :: "r"(row + uint32_t(256 * c + 16 * q)), "f"(v[4 * q]), "f"(v[4 * q + 1]),
                                        "f"(v[4 * q + 2]), "f"(v[4 * q + 3]) : "memory");
                }
                tc::fence_proxy_async();
                bulk_s2g(out + (which == 0 ? OFF_W1 + int64_t(m) * IN + n0 : OFF_W2 + int64_t(m) * HID + n0), row,
                         uint32_t(4 * width));
                bulk_commit();
                bulk_wait();
            }
            tc::fence_before_sync();
        }
    }
    __syncwarp();
    if (threadIdx.x == 128)
        for (int kt = max(0, issued - WG_STAGES); kt < issued; ++kt)
            tc::mbar_wait_bounded(&full[kt % WG_STAGES], (kt / WG_STAGES) & 1, tc::MBAR_SPIN_LIMIT);
    if (threadIdx.x == 160) tc::mbar_wait_bounded(&done, 0, tc::MBAR_SPIN_LIMIT);
    __syncthreads();
    if (threadIdx.x == 0 && *(volatile int*)&fail) atomicOr(err, ERR_TIMEOUT);
    tc::fence_before_sync();
    __syncthreads();
    if (warp == 4) tc::tmem_dealloc(tmem, 512);
}

// ------------------------------------------------------- gradients and update
struct WeightCopies {  // what the tensor cores read
    bf16 *W1, *W2, *W3;   // row-major BF16 (W3 padded to 16 rows)
    bf16 *W2T, *W3T;      // transposed, for the backward pass (W3T: 256 x 64, columns >= 9 zero)
    float* b3p;
};

__device__ __forceinline__ void store_copies(int64_t i, float p, const WeightCopies& w) {
    if (i < OFF_B1) {
        w.W1[i] = __float2bfloat16_rn(p);
    } else if (i >= OFF_W2 && i < OFF_B2) {
        const int j = int(i - OFF_W2);
        const bf16 b = __float2bfloat16_rn(p);
        w.W2[j] = b;
        w.W2T[(j % HID) * HID + j / HID] = b;
    } else if (i >= OFF_W3 && i < OFF_B3) {
        const int j = int(i - OFF_W3);
        const bf16 b = __float2bfloat16_rn(p);
        w.W3[j] = b;
        w.W3T[(j % HID) * DY_STRIDE + j / HID] = b;
    } else if (i >= OFF_B3) {
        w.b3p[i - OFF_B3] = p;
    }
}

// One Adam update; m, v and p are the parameter's moments and value.
__device__ __forceinline__ void adam_one(float g, float& p, float& m, float& v, float lr, float c1, float c2) {
    const float beta1 = 0.9f, beta2 = 0.999f, eps = 1e-8f;
    m = beta1 * m + (1.f - beta1) * g;
    v = beta2 * v + (1.f - beta2) * g * g;
    p -= lr * (m * c1) / (sqrtf(v * c2) + eps);
}

// Gradients from the slices' partials (in slice order) and the column sums
// (in chunk order), and with ADAM the update in the same pass.  Four weights
// per thread; the biases, whose column sums add up in FP64, one per thread of
// the last UPDATE_BIAS_CTAS CTAs (an FP64 warp instruction takes about 64 cycles
// whatever its lanes do: four per thread made them the slowest of the launch).
constexpr int UPDATE_THREADS = 128;
constexpr int UPDATE_BIASES = 2 * HID + OUT;
constexpr int UPDATE_CTAS = int((N_PARAMS + 4 * UPDATE_THREADS - 1) / (4 * UPDATE_THREADS));
constexpr int UPDATE_BIAS_CTAS = (UPDATE_BIASES + UPDATE_THREADS - 1) / UPDATE_THREADS;

template <bool ADAM>
__global__ void __launch_bounds__(UPDATE_THREADS)
k_grad_update(const float* __restrict__ ws, int slices, const float* __restrict__ part, int nchunks,
              float* __restrict__ G, float* __restrict__ P, float* __restrict__ Mo, float* __restrict__ Vo, float lr,
              float c1, float c2, WeightCopies w) {
    if (blockIdx.x >= UPDATE_CTAS) {
        const int b = (int(blockIdx.x) - UPDATE_CTAS) * UPDATE_THREADS + threadIdx.x;
        if (b >= UPDATE_BIASES) return;
        const int mat = b / HID, j = b % HID;
        const int64_t i = (mat == 0 ? OFF_B1 : (mat == 1 ? OFF_B2 : OFF_B3)) + j;
        double s = 0.0;
#pragma unroll 8
        for (int c = 0; c < nchunks; ++c) s += part[(int64_t(c) * 3 + mat) * HID + j];
        const float g = float(s);
        G[i] = g;
        if (ADAM) {
            float p = P[i], m = Mo[i], v = Vo[i];
            adam_one(g, p, m, v, lr, c1, c2);
            Mo[i] = m;
            Vo[i] = v;
            P[i] = p;
            store_copies(i, p, w);
        }
        return;
    }
    const int64_t i0 = 4 * (int64_t(blockIdx.x) * UPDATE_THREADS + threadIdx.x);
    // the biases' ranges start and end on multiples of four
    if (i0 >= OFF_B3 || (i0 >= OFF_B1 && i0 < OFF_W2) || (i0 >= OFF_B2 && i0 < OFF_W3)) return;
    float pv[4], mv[4], vv[4], g[4];
    auto load = [&](const float* src, float (&x)[4]) {
        const float4 t = *reinterpret_cast<const float4*>(src + i0);
        x[0] = t.x;
        x[1] = t.y;
        x[2] = t.z;
        x[3] = t.w;
    };
    auto store = [&](float* dst, const float (&x)[4]) {
        *reinterpret_cast<float4*>(dst + i0) = make_float4(x[0], x[1], x[2], x[3]);
    };
    if (ADAM) {  // in flight with the partials
        load(P, pv);
        load(Mo, mv);
        load(Vo, vv);
    }
    float4 x[WG_MAX_SLICES];
#pragma unroll
    for (int z = 0; z < WG_MAX_SLICES; ++z)
        if (z < slices) x[z] = __ldcg(reinterpret_cast<const float4*>(ws + z * WS_STRIDE + i0));
    g[0] = x[0].x;
    g[1] = x[0].y;
    g[2] = x[0].z;
    g[3] = x[0].w;
#pragma unroll
    for (int z = 1; z < WG_MAX_SLICES; ++z)
        if (z < slices) {
            g[0] += x[z].x;
            g[1] += x[z].y;
            g[2] += x[z].z;
            g[3] += x[z].w;
        }
    store(G, g);
    if (ADAM) {
#pragma unroll
        for (int k = 0; k < 4; ++k) adam_one(g[k], pv[k], mv[k], vv[k], lr, c1, c2);
        store(Mo, mv);
        store(Vo, vv);
        store(P, pv);
        if (i0 < OFF_B1) {
            const __nv_bfloat162 lo = __floats2bfloat162_rn(pv[0], pv[1]), hi = __floats2bfloat162_rn(pv[2], pv[3]);
            *reinterpret_cast<uint2*>(w.W1 + i0) =
                make_uint2(*reinterpret_cast<const uint32_t*>(&lo), *reinterpret_cast<const uint32_t*>(&hi));
        } else {
#pragma unroll
            for (int k = 0; k < 4; ++k) store_copies(i0 + k, pv[k], w);
        }
    }
}

__global__ void k_adam(float* __restrict__ P, const float* __restrict__ G, float* __restrict__ Mo,
                       float* __restrict__ Vo, float lr, float c1, float c2, WeightCopies w) {
    for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < N_PARAMS;
         i += int64_t(gridDim.x) * blockDim.x) {
        float p = P[i], m = Mo[i], v = Vo[i];
        adam_one(G[i], p, m, v, lr, c1, c2);
        Mo[i] = m;
        Vo[i] = v;
        P[i] = p;
        store_copies(i, p, w);
    }
}

__global__ void k_refresh(const float* __restrict__ P, WeightCopies w) {
    for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < N_PARAMS;
         i += int64_t(gridDim.x) * blockDim.x)
        store_copies(i, P[i], w);
}

}  // namespace
}  // namespace hgmm
