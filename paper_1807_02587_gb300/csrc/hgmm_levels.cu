// The build's levels in one cooperative launch, for clouds that the level-wide
// launches of hgmm_build.cu would spend on latency: root statistics, then per
// level the initial children, K EM iterations, the hand-off and the per-node
// eigen-decompositions, with the CTAs meeting through counters instead of
// kernel boundaries.
//
// What bounds it: up to a few hundred thousand points, one EM iteration is
// about a microsecond of arithmetic; the launches spent 7.5 us on an E-step
// and 10 us on an M-step (93k points), nearly all of it launch, load and
// reduction latency.  So
//   - every CTA keeps its points (one contiguous range, at most LV_MAX_RUNS
//     runs of at most LV_RUN_POINTS points of one parent) in shared memory for
//     all iterations of a level, the hand-off included;
//   - a run sums at most 16 points per lane in plain FP32, so its moments need
//     exactly one compensated fold and no running (sum, error) pairs;
//   - CTAs wait only for the runs of their own parents (one arrival counter
//     per parent), and every CTA that holds a run of a parent reduces that
//     parent's runs and computes its M-step itself, in the same order on the
//     same values (so all get the same bits): the new parameters need no
//     second round trip.  A parent of more than LV_DIRECT_RUNS runs is reduced
//     in slices of LV_SLICE_RUNS runs by as many CTAs first (one more hop,
//     but no CTA reads hundreds of partials);
//   - the eigen-decompositions of a parent's children run on one warp beside
//     the hand-off of the points.
// The runs are those of the level-wide launches (chunks of C items per CTA of
// the E-step grid; from LOCAL_EM_PARENTS parents up, groups of four items of a
// parent), so the plain FP32 sums hold the same points in the same order.  The
// compensated sums over runs (and over the root's partials) group them
// otherwise, so the two builds' records agree to about 1e-14 (relative), not to
// the last bit.
//
// Measured (one GB300; kernel time of the whole build): 93k LiDAR points, depth
// 4: 815 us in 76 launches before, 501 us here; per EM iteration 17.6 us before
// against 11.9 (level 0: E-step 1.8, publishing 0.8, slices 3.7, waiting 1.2,
// reduction 1.2, M-step 3.4), 10.5, 8.2 and 6.0 at levels 1, 2 and 3.
//
// All waits are bounded: a wait that runs out records ST_TIMEOUT and the CTA
// returns (the others then run out too).
#include <algorithm>
#include <cstdio>

#include "hgmm_dev.cuh"
#include "hgmm_levels.cuh"

namespace hgmm {

namespace {

constexpr int LV_THREADS = EST_THREADS;
constexpr int LV_MAX_RUNS = 4;                      // runs (and parents) of a CTA at one level
constexpr int LV_RUN_ITEMS = 4;
constexpr int LV_RUN_POINTS = LV_RUN_ITEMS * TILE;  // EST_FOLD steps of 64 points
constexpr int LV_LOCAL_UNITS = 2;                   // runs per CTA of a level with many parents
constexpr int LV_MAX_LEVELS = 4;                    // levels this launch can run (512 parents)
constexpr int LV_MAX_PARENTS = 512;
constexpr int LV_DIRECT_RUNS = 32;
constexpr int LV_SLICE_RUNS = 24;
constexpr int LV_CNT = 1 + 8 + 64 + 512;            // parents of all levels
static_assert(LV_RUN_POINTS == 64 * EST_FOLD, "a run is one compensated fold");
static_assert(LV_THREADS == 256, "eight warps");

struct LvRun {
    int par;     // local parent index
    int off;     // first point, from the CTA's first
    int count;   // points
    int slot;    // first item: the run's partial
    int j;       // index of the run within its parent
};

struct LvPar {
    int p;       // parent index within the level
    int item0;   // its first item
    int items;
    int nruns;
    int rbase, rstride;  // run j > 0 starts at item rbase + j * rstride
    int seg;     // segment start
    int count;   // its points
    int owner;   // this CTA holds its first run
};

struct LvSmem {
    int item0[LV_MAX_PARENTS + 1];
    int unit0[LV_MAX_PARENTS + 1];
    LvRun run[LV_MAX_RUNS];
    LvPar par[LV_MAX_RUNS];
    int n_runs, n_par, first, total;
    RootDev root;
    alignas(16) NodeEst est[LV_MAX_RUNS][8];
    int live[LV_MAX_RUNS][8];
    double mom[LV_MAX_RUNS][NPART];
    union {
        float2 red[LV_MAX_RUNS][EST_THREADS / 32][NPART];
        RootSmem rs;
        struct {
            int cnt[2 * LV_RUN_ITEMS][EST_THREADS / 32][8];  // per item and warp: points per child
            int sum[EST_THREADS / 32][2][8];
            int base[2 * LV_RUN_ITEMS][8];
            uint16_t code[2 * LV_RUN_POINTS];
            int scan[33];
        };
    };
};

__device__ __forceinline__ bool poll_at_least(const unsigned* word, unsigned target, int* status) {
    unsigned v;
    for (long long spins = 0;; ++spins) {
        asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(word) : "memory");
        if (int(v - target) >= 0) break;
        if (spins > BARRIER_SPIN_LIMIT) {
            atomicOr(status, ST_TIMEOUT);
            return false;
        }
    }
    asm volatile("fence.acq_rel.gpu;" ::: "memory");
    return true;
}

// The whole grid meets (counter zeroed before the launch; `target` = barriers
// so far x grid).  Every earlier global write of the grid is visible after it.
__device__ __forceinline__ bool lv_grid_sync(unsigned* bar, unsigned target, int* status) {
    __syncthreads();
    bool ok = true;
    if (threadIdx.x == 0) {
        arrive_release(bar);
        ok = poll_at_least(bar, target, status);
    }
    return !__syncthreads_or(!ok);
}

// The first level of flush_run's reduce-scatter for sums without an error yet.
__device__ __forceinline__ void flush_rs_first(float (&s)[20], float (&c)[20], int lane) {
    const bool up = (lane & 16) != 0;
#pragma unroll
    for (int i = 0; i < 10; ++i) {
        const float sr = __shfl_xor_sync(FULL, up ? s[i] : s[10 + i], 16);
        const float sk = up ? s[10 + i] : s[i];
        two_sum(sk, sr, s[i], c[i]);
    }
}

// Slot of run j of a parent (in items).
__device__ __forceinline__ int run_slot(const LvPar& q, int j) { return j == 0 ? q.item0 : q.rbase + j * q.rstride; }

// Sums of `rows` (at most 32) rows of NPART pairs into sm.red[i][warp], four rows a warp.
template <class Row>
__device__ __forceinline__ void reduce_rows(int rows, Row row, float2 (*red)[NPART]) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    float2 x[4][3];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const int r = warp + 8 * u;
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            const int v = lane + 32 * q;
            x[u][q] = (r < rows && v < NPART) ? __ldcg(row(r) + v) : make_float2(0.f, 0.f);
        }
    }
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        const int v = lane + 32 * q;
        float S = x[0][q].x, C = x[0][q].y;
#pragma unroll
        for (int u = 1; u < 4; ++u) pair_add(S, C, x[u][q].x, x[u][q].y);
        if (v < NPART) red[warp][v] = make_float2(S, C);
    }
}

__device__ __forceinline__ float2 sum_warps(const float2 (*red)[NPART], int v) {
    float S = 0.f, C = 0.f;
#pragma unroll
    for (int w = 0; w < EST_THREADS / 32; ++w) pair_add(S, C, red[w][v].x, red[w][v].y);
    return make_float2(S, C);
}

__device__ __forceinline__ void bar_lower() { asm volatile("bar.sync 1, 128;" ::: "memory"); }

// This CTA's runs and parents of a level (thread 0), from the item (and run)
// prefixes in shared memory.
__device__ void lv_find_runs(LvSmem& sm, int n_par, bool local, int n_chunks) {
    const int items = sm.item0[n_par];
    int nr = 0, np = 0;
    auto parent_of = [&](const int* pre, int x) {  // the last parent that starts at or before x
        int lo = 0, hi = n_par - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (pre[mid] <= x) lo = mid;
            else hi = mid - 1;
        }
        return lo;
    };
    auto add = [&](int p, int first_item, int n_items, int j, int rbase, int rstride, int nruns) {
        if (np == 0 || sm.par[np - 1].p != p) {
            LvPar& q = sm.par[np++];
            q.p = p;
            q.item0 = sm.item0[p];
            q.items = sm.item0[p + 1] - sm.item0[p];
            q.nruns = nruns;
            q.rbase = rbase;
            q.rstride = rstride;
            q.owner = 0;
        }
        if (j == 0) sm.par[np - 1].owner = 1;
        LvRun& r = sm.run[nr++];
        r.par = np - 1;
        r.slot = first_item;
        r.count = n_items;  // items for now
        r.j = j;
    };
    if (local) {
        const int units = sm.unit0[n_par];
        const int U = max(1, (units + int(gridDim.x) - 1) / int(gridDim.x));
        const int ub = blockIdx.x * U, ue = min(ub + U, units);
        if (ub < ue && U <= LV_LOCAL_UNITS) {
            int p = parent_of(sm.unit0, ub);
            for (int u = ub; u < ue; ++u) {
                while (sm.unit0[p + 1] <= u) ++p;
                const int j = u - sm.unit0[p], it = sm.item0[p] + LV_RUN_ITEMS * j;
                add(p, it, min(LV_RUN_ITEMS, sm.item0[p + 1] - it), j, sm.item0[p], LV_RUN_ITEMS,
                    sm.unit0[p + 1] - sm.unit0[p]);
            }
        }
    } else {
        const int C = max(1, (items + n_chunks - 1) / n_chunks);
        const int ib = blockIdx.x * C, ie = min(ib + C, items);
        if (ib < ie && C <= LV_RUN_ITEMS) {
            int p = parent_of(sm.item0, ib);
            for (int it = ib; it < ie;) {
                while (sm.item0[p + 1] <= it) ++p;
                const int e = min(ie, sm.item0[p + 1]);
                const int b0 = sm.item0[p] / C;
                add(p, it, e - it, int(blockIdx.x) - b0, b0 * C, C, (sm.item0[p + 1] - 1) / C - b0 + 1);
                it = e;
            }
        }
    }
    sm.n_runs = nr;
    sm.n_par = np;
}

__global__ void __launch_bounds__(LV_THREADS, LV_CTAS_PER_SM) k_build_levels(LevelsArgs a) {
    __shared__ LvSmem sm;
    extern __shared__ float4 spts[];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int cta = blockIdx.x, ncta = gridDim.x;
    unsigned* const bar = a.cnt;
    unsigned* const arrivals = a.cnt + 1;             // per parent of every level: its runs
    unsigned* const sliced = a.cnt + 1 + LV_CNT;      // ... its slices
    unsigned barriers = 0;

    // ---- root: every CTA reduces the partials itself
    root_partial_cta(a.pts, a.n, cta, ncta, a.root_part + 32 * cta, sm.rs);
    if (!lv_grid_sync(bar, ++barriers * unsigned(ncta), a.status)) return;
    root_final_cta(a.root_part, ncta, a.pts, a.n, a.eps_rel, &sm.root, cta == 0 ? a.status : nullptr, sm.rs);
    if (cta == 0) {
        const double* s = reinterpret_cast<const double*>(&sm.root);
        for (int i = tid; i < int(sizeof(RootDev) / 8); i += LV_THREADS) reinterpret_cast<double*>(a.root)[i] = s[i];
    }
    const double eps = sm.root.eps;
    const float4* cur = a.pts;
    const int* perm_in = nullptr;
    int pbase = 0;  // first counter of the level's parents
    for (int l = 0; l < a.levels; ++l) {
        const int n_par = l == 0 ? 1 : 1 << (3 * l);
        const int poff = l == 0 ? 0 : int(d_level_offset(l - 1));  // first parent's node
        const int coff = int(d_level_offset(l));                   // first child's node
        const bool local = n_par >= LOCAL_EM_PARENTS;
        const bool stop_here = a.stop_level == l + 1;
        const int K = stop_here ? a.stop_iters : a.em_iters;
        // ---- items and runs of every parent (exclusive prefixes; every CTA for itself)
        {
            int x[2], inc = 0;  // runs << 16 | items of this thread's two parents
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int p = 2 * tid + h;
                const int count = p < n_par ? (l == 0 ? a.n : __ldcg(a.seg_count + poff + p)) : 0;
                const int k = (count + TILE - 1) / TILE;
                x[h] = k | ((k + LV_RUN_ITEMS - 1) / LV_RUN_ITEMS) << 16;
                inc += x[h];
            }
            int w = inc;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(FULL, w, o);
                if (lane >= o) w += y;
            }
            if (lane == 31) sm.scan[warp] = w;
            __syncthreads();
            int ex = w - inc;
            for (int q = 0; q < warp; ++q) ex += sm.scan[q];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int p = 2 * tid + h;
                if (p <= n_par) {
                    sm.item0[p] = ex & 0xFFFF;
                    sm.unit0[p] = ex >> 16;
                }
                ex += x[h];
            }
            if (tid == LV_THREADS - 1 && n_par == 2 * LV_THREADS) {
                sm.item0[n_par] = ex & 0xFFFF;
                sm.unit0[n_par] = ex >> 16;
            }
        }
        __syncthreads();
        if (tid == 0) lv_find_runs(sm, n_par, local, a.n_chunks);
        __syncthreads();
        const int nr = sm.n_runs, np = sm.n_par;
        if (tid < np) {
            LvPar& q = sm.par[tid];
            q.seg = l == 0 ? 0 : __ldcg(a.seg_start + poff + q.p);
            q.count = l == 0 ? a.n : __ldcg(a.seg_count + poff + q.p);
        }
        __syncthreads();
        if (tid < nr) {  // the runs' points: one contiguous range
            LvRun& r = sm.run[tid];
            const LvPar& q = sm.par[r.par];
            const int in_par = (r.slot - q.item0) * TILE;
            const LvRun& r0 = sm.run[0];
            const int first = sm.par[r0.par].seg + (r0.slot - sm.par[r0.par].item0) * TILE;
            r.off = q.seg + in_par - first;
            const int cnt = min(r.count * TILE, q.count - in_par);
            __syncwarp((1u << nr) - 1u);
            r.count = cnt;
            if (tid == 0) sm.first = first;
            if (tid == nr - 1) sm.total = r.off + cnt;
        }
        __syncthreads();
        const int first = nr ? sm.first : 0, total = nr ? sm.total : 0;
        for (int i = tid; i < total; i += LV_THREADS) spts[i] = __ldcg(cur + first + i);
        // ---- initial children: one warp per parent of this CTA; parents
        // without points (dead children) dealt over the CTAs' upper warps
        if (warp < np) {
            const LvPar& q = sm.par[warp];
            if (lane < 8) {
                double lam[3], V[9], mu[3], S[6];
                bool alive = true;
                if (l == 0) {
                    for (int v = 0; v < 3; ++v) { mu[v] = sm.root.mu[v]; lam[v] = sm.root.lam[v]; }
                    for (int v = 0; v < 6; ++v) S[v] = sm.root.S[v];
                    for (int v = 0; v < 9; ++v) V[v] = sm.root.V[v];
                } else {
                    const NodeStat* ps = a.stat + poff + q.p;
                    for (int v = 0; v < 3; ++v) { mu[v] = __ldcg(ps->mu + v); lam[v] = __ldcg(ps->lam + v); }
                    for (int v = 0; v < 6; ++v) S[v] = __ldcg(ps->S + v);
                    for (int v = 0; v < 9; ++v) V[v] = __ldcg(ps->V + v);
                    alive = __ldcg(&ps->live) != 0 && q.count > 0;
                }
                const int64_t g = coff + 8 * int64_t(q.p) + lane;
                NodeEst& e = sm.est[warp][lane];
                init_child_of(alive, mu, S, lam, V, eps, lane, q.owner ? a.stat + g : nullptr, e, a.status);
                sm.live[warp][lane] = alive;
                if (q.owner) a.est[g] = e;
            }
        } else if (warp >= LV_MAX_RUNS && l > 0) {
            for (int p = cta + ncta * (warp - LV_MAX_RUNS); p < n_par; p += ncta * LV_MAX_RUNS) {
                if (sm.item0[p] != sm.item0[p + 1] || lane >= 8) continue;
                const NodeStat* ps = a.stat + poff + p;
                const double mu[3] = {__ldcg(ps->mu), __ldcg(ps->mu + 1), __ldcg(ps->mu + 2)};
                const double z3[3] = {}, z6[6] = {}, z9[9] = {};
                const int64_t g = coff + 8 * int64_t(p) + lane;
                init_child_of(false, mu, z6, z3, z9, eps, lane, a.stat + g, a.est[g], a.status);
            }
        }
        __syncthreads();

        // ---- K EM iterations
        for (int k = 0; k < K && nr > 0; ++k) {
            float2* const part = a.part + (k & 1) * a.part_stride;
            float2* const slices = a.slices + (k & 1) * a.slice_stride;
            for (int r = 0; r < nr; ++r) {
                const LvRun rn = sm.run[r];
                ChildPair cp;
                load_child_pair(sm.est[rn.par] + 2 * (lane & 3), cp);
                float2 in[10];
#pragma unroll
                for (int v = 0; v < 10; ++v) in[v] = make_float2(0.f, 0.f);
                if (parent_has_live_child(cp)) {  // else zero posteriors: nothing to add
                    const float4* z = spts + rn.off;
                    for (int i = warp * 8 + (lane >> 2); i - (lane >> 2) - warp * 8 < rn.count; i += 64)
                        estep_point_pair(cp, z[min(i, rn.count - 1)], i < rn.count, in);
                }
                float s[20], c[20];
#pragma unroll
                for (int v = 0; v < 10; ++v) {
                    s[v] = in[v].x;
                    s[10 + v] = in[v].y;
                }
                flush_rs_first(s, c, lane);
                flush_rs_level<true, 10, 8>(s, c, lane);
                flush_rs_level<true, 5, 4>(s, c, lane);
                const int base = ((lane & 16) ? 10 : 0) + ((lane & 8) ? 5 : 0) + ((lane & 4) ? 3 : 0);
                const int cnt = (lane & 4) ? 2 : 3;
#pragma unroll
                for (int i = 0; i < 3; ++i)
                    if (i < cnt) sm.red[r][warp][(lane & 3) * 20 + base + i] = make_float2(s[i], c[i]);
            }
            __syncthreads();
            for (int i = tid; i < nr * NPART; i += LV_THREADS) {
                const int r = i / NPART, v = i - r * NPART;
                const float2 x = sum_warps(sm.red[r], v);
                const LvRun& rn = sm.run[r];
                if (sm.par[rn.par].nruns == 1) sm.mom[rn.par][v] = double(x.x) + double(x.y);
                else part[int64_t(rn.slot) * NPART + v] = x;
            }
            __syncthreads();
            bool ok = true;
            if (tid < nr) {
                const LvPar& q = sm.par[sm.run[tid].par];
                if (q.nruns > 1) arrive_release(arrivals + pbase + q.p);
            }
            // slices of parents with many runs
            for (int r = 0; r < nr; ++r) {
                const LvRun& rn = sm.run[r];
                const LvPar& q = sm.par[rn.par];
                const int ns = (q.nruns + LV_SLICE_RUNS - 1) / LV_SLICE_RUNS;
                if (q.nruns <= LV_DIRECT_RUNS || rn.j >= ns) continue;  // uniform over the CTA
                if (tid == 0) ok = poll_at_least(arrivals + pbase + q.p, unsigned(k + 1) * unsigned(q.nruns), a.status);
                if (__syncthreads_or(!ok)) return;
                const int j0 = rn.j * LV_SLICE_RUNS;
                reduce_rows(min(LV_SLICE_RUNS, q.nruns - j0),
                            [&](int x) { return part + int64_t(run_slot(q, j0 + x)) * NPART; }, sm.red[0]);
                __syncthreads();
                if (tid < NPART) slices[int64_t(q.item0 / 8 + rn.j) * NPART + tid] = sum_warps(sm.red[0], tid);
                __syncthreads();
                if (tid == 0) arrive_release(sliced + pbase + q.p);
            }
            // every parent's runs (or slices), reduced by each CTA that holds one of its runs
            if (tid < np) {
                const LvPar& q = sm.par[tid];
                const int ns = (q.nruns + LV_SLICE_RUNS - 1) / LV_SLICE_RUNS;
                if (q.nruns > LV_DIRECT_RUNS)
                    ok = poll_at_least(sliced + pbase + q.p, unsigned(k + 1) * unsigned(ns), a.status);
                else if (q.nruns > 1)
                    ok = poll_at_least(arrivals + pbase + q.p, unsigned(k + 1) * unsigned(q.nruns), a.status);
            }
            if (__syncthreads_or(!ok)) return;
            for (int i = 0; i < np; ++i) {
                const LvPar& q = sm.par[i];
                if (q.nruns > LV_DIRECT_RUNS)
                    reduce_rows((q.nruns + LV_SLICE_RUNS - 1) / LV_SLICE_RUNS,
                                [&](int x) { return slices + int64_t(q.item0 / 8 + x) * NPART; }, sm.red[i]);
                else if (q.nruns > 1)
                    reduce_rows(q.nruns, [&](int x) { return part + int64_t(run_slot(q, x)) * NPART; }, sm.red[i]);
            }
            __syncthreads();
            for (int t = tid; t < np * NPART; t += LV_THREADS) {
                const int i = t / NPART, v = t - i * NPART;
                if (sm.par[i].nruns > 1) {
                    const float2 x = sum_warps(sm.red[i], v);
                    sm.mom[i][v] = double(x.x) + double(x.y);
                }
            }
            __syncthreads();
            if (warp < np) {
                const LvPar& q = sm.par[warp];
                const int64_t g0 = coff + 8 * int64_t(q.p);
                const bool live = child_mstep_at(double(q.count), sm.mom[warp], eps, a.n_min,
                                                 sm.live[warp][lane >> 2] != 0, sm.est[warp],
                                                 q.owner ? a.stat + g0 : nullptr, q.owner ? a.est + g0 : nullptr,
                                                 a.status);
                __syncwarp();
                if ((lane & 3) == 0) sm.live[warp][lane >> 2] = live;
            }
            __syncthreads();
        }
        if (stop_here) return;  // checking aid: parameters after K iterations

        // ---- hand-off: argmax child of every point (ties to the lowest
        // index) and its rank among the item's points of that child
        const bool dead_work = l > 0;
        int it_of[LV_MAX_RUNS + 1];  // local items before each run
        it_of[0] = 0;
#pragma unroll
        for (int r = 0; r < LV_MAX_RUNS; ++r)
            it_of[r + 1] = it_of[r] + (r < nr ? (sm.run[r].count + TILE - 1) / TILE : 0);
        for (int r = 0; r < nr; ++r) {
            const LvRun rn = sm.run[r];
            for (int b = 0; b < rn.count; b += TILE) {
                const int i = b + tid;
                const bool valid = i < rn.count;
                const float4 z = spts[rn.off + min(i, rn.count - 1)];
                int lab = 0;
                float best = 0.f;
#pragma unroll
                for (int c = 0; c < 8; ++c) {
                    ChildRegs cr;
                    load_child(sm.est[rn.par] + c, cr);
                    float ex, ey, ez;
                    const float sc = child_score(cr, z.x, z.y, z.z, ex, ey, ez);
                    if (c == 0 || sc > best) {
                        best = sc;
                        lab = c;
                    }
                }
                const int it = it_of[r] + b / TILE;
                int rank = 0;
#pragma unroll
                for (int c = 0; c < 8; ++c) {
                    const unsigned m = __ballot_sync(FULL, valid && lab == c);
                    if (lab == c) rank = __popc(m & ((1u << lane) - 1u));
                    if (lane == c) sm.cnt[it][warp][c] = __popc(m);
                }
                if (valid) sm.code[rn.off + i] = uint16_t(lab | rank << 3);
            }
        }
        __syncthreads();
        // the items' child counts; a count per warp becomes the warps before it
        const int n_it = it_of[LV_MAX_RUNS];
        if (tid < 8 * n_it) {
            const int it = tid >> 3, c = tid & 7;
            int s = 0;
#pragma unroll
            for (int w = 0; w < EST_THREADS / 32; ++w) {
                const int x = sm.cnt[it][w][c];
                sm.cnt[it][w][c] = s;
                s += x;
            }
            int r = 0;
            while (r + 1 < nr && it >= it_of[r + 1]) ++r;
            a.item_cnt[8 * (sm.run[r].slot + it - it_of[r]) + c] = s;
            sm.base[it][c] = s;  // the item's own counts, until its offsets replace them
        }
        __syncthreads();
        if (tid < nr) {
            const LvPar& q = sm.par[sm.run[tid].par];
            if (q.nruns > 1) arrive_release(arrivals + pbase + q.p);
        }
        float4* const out = a.buf[l & 1];
        int* const perm_out = a.perm[l];
        bool ok = true;
        if (warp < 4) {
            // destinations: the parent's start, its children before, its items before
            if (tid < np) {
                const LvPar& q = sm.par[tid];
                if (q.nruns > 1)
                    ok = poll_at_least(arrivals + pbase + q.p, unsigned(K + 1) * unsigned(q.nruns), a.status);
            }
            bar_lower();
            for (int r = 0; r < nr; ++r) {
                const LvRun rn = sm.run[r];
                const LvPar& q = sm.par[rn.par];
                int tot = 0, pre = 0;  // of child tid & 7, over items q.item0 + (tid >> 3) + 16 k
                const int c = tid & 7;
#pragma unroll 8
                for (int i = tid >> 3; i < q.items; i += 16) {
                    const int x = __ldcg(a.item_cnt + 8 * (q.item0 + i) + c);
                    tot += x;
                    pre += q.item0 + i < rn.slot ? x : 0;
                }
#pragma unroll
                for (int o = 8; o < 32; o <<= 1) {
                    tot += __shfl_xor_sync(FULL, tot, o);
                    pre += __shfl_xor_sync(FULL, pre, o);
                }
                if (lane < 8) {
                    sm.sum[warp][0][c] = tot;
                    sm.sum[warp][1][c] = pre;
                }
                bar_lower();
                if (tid < 8) {
                    int run = 0, before = 0;
                    for (int w = 0; w < 4; ++w) {
                        run += sm.sum[w][0][c];
                        before += sm.sum[w][1][c];
                    }
                    int inc = run;
#pragma unroll
                    for (int o = 1; o < 8; o <<= 1) {
                        const int y = __shfl_up_sync(0xFFu, inc, o);
                        if (lane >= o) inc += y;
                    }
                    const int start = q.seg + inc - run;
                    if (rn.j == 0) {
                        a.seg_start[coff + 8 * q.p + c] = start;
                        a.seg_count[coff + 8 * q.p + c] = run;
                    }
                    int at = start + before;
                    const int n_items = (rn.count + TILE - 1) / TILE;
                    for (int i = 0; i < n_items; ++i) {
                        const int x = sm.base[it_of[r] + i][c];
                        sm.base[it_of[r] + i][c] = at;
                        at += x;
                    }
                }
                bar_lower();
                for (int i = tid; i < rn.count; i += 128) {
                    const int code = sm.code[rn.off + i], lab = code & 7, it = it_of[r] + i / TILE;
                    const int dst = sm.base[it][lab] + sm.cnt[it][(i & (TILE - 1)) >> 5][lab] + (code >> 3);
                    const int pos = first + rn.off + i;
                    if (unsigned(dst) < unsigned(a.n)) {  // always, unless a wait ran out
                        out[dst] = spts[rn.off + i];
                        perm_out[dst] = perm_in ? __ldcg(perm_in + pos) : pos;
                    }
                }
            }
        } else {
            // finalise the children of the parents this CTA owns, and of its share of the empty ones
            const int i = warp - 4;
            if (i < np && sm.par[i].owner && lane < 8)
                finalize_node(l, 8 * int64_t(sm.par[i].p) + lane, a.lam_c, &sm.root, a.stat, a.est, a.rnode);
            if (dead_work)
                for (int p = cta + ncta * i; p < n_par; p += ncta * 4) {
                    if (sm.item0[p] != sm.item0[p + 1] || lane >= 8) continue;
                    const int64_t g = coff + 8 * int64_t(p) + lane;
                    a.seg_start[g] = __ldcg(a.seg_start + poff + p);
                    a.seg_count[g] = 0;
                    finalize_node(l, 8 * int64_t(p) + lane, a.lam_c, &sm.root, a.stat, a.est, a.rnode);
                }
        }
        if (__syncthreads_or(!ok)) return;
        cur = out;
        perm_in = perm_out;
        pbase += n_par;
        if (l + 1 < a.levels && !lv_grid_sync(bar, ++barriers * unsigned(ncta), a.status)) return;
    }
}

}  // namespace

// Items of the deepest level the launch can run (the partials' slots).
int64_t levels_slots(int64_t n) { return (n + TILE - 1) / TILE + LV_MAX_PARENTS; }

int levels_counters() { return 1 + 2 * LV_CNT; }

bool levels_smem_attr() {
    int k = 0;
    return cudaFuncSetAttribute(k_build_levels, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                LV_LOCAL_UNITS * LV_RUN_POINTS * int(sizeof(float4))) == cudaSuccess &&
           cudaOccupancyMaxActiveBlocksPerMultiprocessor(&k, k_build_levels, LV_THREADS,
                                                         LV_LOCAL_UNITS * LV_RUN_POINTS * sizeof(float4)) ==
               cudaSuccess &&
           k >= LV_CTAS_PER_SM;
}

// Levels of an n-point, depth-level build that the launch takes (0: none).
// Its CTAs must hold every point of a level: at most LV_RUN_ITEMS items per
// chunk, and LV_LOCAL_UNITS runs per CTA where a level has many parents.  Up to
// that capacity it is the faster one at every size: depth-4 builds of 100k /
// 277k / 400k points take 517 / 591 / 673 us against 797 / 948 / 981 with the
// level-wide launches, depth-3 builds of 1k / 10k points 242 / 287 against
// 529 / 554.
int levels_taken(int64_t n, int depth, int est_grid) {
    const int L = std::min(depth, LV_MAX_LEVELS);
    const int64_t items = (n + TILE - 1) / TILE;
    for (int l = 0; l < L; ++l) {
        const int64_t n_par = l == 0 ? 1 : level_size(l - 1);
        if (n_par >= LOCAL_EM_PARENTS) {
            if (n > LOCAL_EM_POINTS * n_par ||
                n / LV_RUN_POINTS + n_par > int64_t(LV_LOCAL_UNITS) * est_grid)
                return 0;
        } else if (items + n_par > int64_t(LV_RUN_ITEMS) * est_grid) {
            return 0;
        }
    }
    return L;
}

int levels_launch(LevelsArgs& a, int est_grid, bool refuse, cudaStream_t s) {
    // CTAs: as many as a level has chunks or runs, at most the E-step's grid
    // (a barrier of fewer CTAs is cheaper); one chunk of the level-wide
    // launches per CTA
    const int64_t items = (a.n + TILE - 1) / TILE;
    int64_t want = 1;
    bool many = false;
    for (int l = 0; l < a.levels; ++l) {
        const int64_t n_par = l == 0 ? 1 : level_size(l - 1);
        const bool local = n_par >= LOCAL_EM_PARENTS;
        many = many || local;
        want = std::max(want, local ? a.n / LV_RUN_POINTS + n_par : items + n_par - 1);
    }
    const int grid = refuse ? 64 * est_grid : int(std::min<int64_t>(want, est_grid));
    a.n_chunks = est_grid;
    if (cudaMemsetAsync(a.cnt, 0, size_t(levels_counters()) * sizeof(unsigned), s) != cudaSuccess) return HGMM_ECUDA;
    void* args[] = {&a};
    const size_t smem = (many ? LV_LOCAL_UNITS : 1) * LV_RUN_POINTS * sizeof(float4);
    const cudaError_t e =
        cudaLaunchCooperativeKernel((const void*)k_build_levels, dim3(grid), dim3(LV_THREADS), args, smem, s);
    if (e == cudaErrorCooperativeLaunchTooLarge || e == cudaErrorLaunchOutOfResources || e == cudaErrorNotSupported) {
        cudaGetLastError();
        return LEVELS_REFUSED;
    }
    if (e != cudaSuccess) {
        fprintf(stderr, "hgmm: cooperative build launch failed: %s\n", cudaGetErrorString(cudaGetLastError()));
        return HGMM_ECUDA;
    }
    return HGMM_OK;
}

}  // namespace hgmm
