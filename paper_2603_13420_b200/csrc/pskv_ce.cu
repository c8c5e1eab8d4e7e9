// Masked target cross-entropy fused with the vocabulary projection, for sm_100a (tcgen05 / TMEM / TMA).
//
// logits = hidden * weight^T is a [rows x V] matrix that is only ever reduced: per row its
// log-sum-exp and the logit of the target token (loss appendix: masked average of CE over the
// target-response span).  Forming it in memory is what the paper names as the memory high-water
// mark of a search step, so here it never leaves the chip: a 128-row x 256-column block of logits is
// accumulated in tensor memory over the hidden dimension, four warps fold it into a running
// (max, sum) per row and pick out the target's logit while the tensor cores already work on the next
// block in the other half of tensor memory.
//
// Work units are (vocabulary panel of up to 16 blocks, 128-row tile); the panel is as wide as lets the units
// fill whole rounds of the SMs (ce_panel).  Row tiles are taken in groups of a
// quarter of the CTA count; inside a group the units are numbered panel-major, row tile fastest, and
// CTA c takes units c, c + G, c + 2G, ...: the CTAs running at any moment work on about four weight
// panels (16 MB each) against one group of row tiles (1 MB each), a working set that stays in L2, so
// the weight matrix comes from HBM once per row group and the hidden states once.  Each unit
// leaves one partial (max, sum) per row; a small kernel merges the partials of a row into lse and nll = mask * (lse -
// target logit) and forms the masked average of each candidate (with many rows per candidate a second one does).
//
// Roles (256 threads): warp 0 TMA producer (hidden tile and weight block, 64 columns of the hidden
// dimension per stage, 4 stages), warp 1 tcgen05.mma issuer, warp 2 owns the tensor-memory
// allocation, warps 4-7 fold the finished blocks.  Every wait is bounded.
#include <string.h>

#include "pskv_common.cuh"
#include "pskv_sm100.cuh"
#include "pskv_tc_common.cuh"

namespace pskv {
namespace {

using namespace sm100;

constexpr int kCeM = 128;        // rows per tile (tensor-memory lanes)
constexpr int kCeN = 256;        // vocabulary entries per block (one MMA N, half of tensor memory)
constexpr int kCeK = 64;         // hidden columns per stage: one 128-byte swizzle slab
constexpr int kCeStages = 4;
constexpr int kCeMaxPanel = 16;  // blocks per panel at most
constexpr int kCeThreads = 256;
constexpr int kCeABytes = kCeM * 128, kCeBBytes = kCeN * 128, kCeStageBytes = kCeABytes + kCeBBytes;

enum : unsigned int { kErrCeProducer = 0x401, kErrCeMma = 0x402, kErrCeFold = 0x403, kErrCeAlign = 0x404 };

enum { kCeBarFull = 0, kCeBarEmpty = kCeStages, kCeBarAccFull = 2 * kCeStages, kCeBarAccFree = 2 * kCeStages + 2,
       kCeNumBars = 2 * kCeStages + 4 };

struct CeParams {
    const int *target;     // [R]
    float2 *part;          // [R][npanel] (max, sum), log2 domain
    float *tlogit;         // [R] logit of the target token (natural units)
    unsigned int *status;
    int R, Dm, V;
    int nrt, nvb, panel, npanel, units, ksteps;
    int rg;                // row tiles per group
};

// unit -> (panel, row tile): groups of rg row tiles, panel-major inside a group, the last group smaller
__device__ __forceinline__ void ce_unit(const CeParams &p, int u, int &pn, int &rt)
{
    const int per_group = p.rg * p.npanel;
    const int nfull = p.nrt / p.rg;
    if (u < nfull * per_group) {
        const int gi = u / per_group, rem = u - gi * per_group;
        pn = rem / p.rg;
        rt = gi * p.rg + (rem - pn * p.rg);
    } else {
        const int tail = p.nrt - nfull * p.rg, rem = u - nfull * per_group;
        pn = rem / tail;
        rt = nfull * p.rg + (rem - pn * tail);
    }
}

__global__ void __launch_bounds__(kCeThreads, 1)
ce_fwd_kernel(const __grid_constant__ CUtensorMap tm_h, const __grid_constant__ CUtensorMap tm_w, const CeParams p)
{
    extern __shared__ __align__(1024) uint8_t smem[];
    const int tid = threadIdx.x, lane = tid & 31;
    const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
    const uint32_t sbase = smem_u32(smem);
    const uint32_t bar0 = sbase + kCeStages * kCeStageBytes;
    auto bar = [&](int i) { return bar0 + 8u * (uint32_t)i; };
    volatile int *abort_flag = reinterpret_cast<volatile int *>(smem + kCeStages * kCeStageBytes + 8 * kCeNumBars + 4);
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(smem + kCeStages * kCeStageBytes + 8 * kCeNumBars);

    if ((sbase & 1023u) != 0u) {
        if (tid == 0) atomicCAS(p.status, 0u, (unsigned int)kErrCeAlign);
        return;
    }
    if (tid == 0) {
        for (int i = 0; i < kCeNumBars; ++i) mbar_init(bar(i), i >= kCeBarAccFree ? 4u : 1u);
        *abort_flag = 0;
        fence_barrier_init();
    }
    __syncthreads();
    if (warp == 2) {
        tmem_alloc(smem_u32(tmem_slot), 512);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    const int n_units = (p.units - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x;

    if (warp == 0) {
        // ------------------------------------------------------------------ TMA producer
        if (lane == 0) {
            prefetch_tensormap(&tm_h);
            prefetch_tensormap(&tm_w);
        }
        uint32_t it = 0;
        bool ok = true;
#pragma unroll 1
        for (int tl = 0; tl < n_units && ok; ++tl) {
            const int u = (int)blockIdx.x + tl * (int)gridDim.x;
            int pn, rt;
            ce_unit(p, u, pn, rt);
            const int vb_end = min(p.nvb, (pn + 1) * p.panel);
#pragma unroll 1
            for (int vb = pn * p.panel; vb < vb_end && ok; ++vb) {
#pragma unroll 1
                for (int ks = 0; ks < p.ksteps; ++ks, ++it) {
                    const uint32_t s = it % kCeStages;
                    ok = mbar_wait_warp(bar(kCeBarEmpty + s), ((it / kCeStages) & 1) ^ 1, abort_flag, p.status,
                                        kErrCeProducer);
                    if (!ok) break;
                    if (elect_one_sync()) {
                        // boxes that reach past the last row / vocabulary entry / hidden column are
                        // zero-filled and still count their full size
                        mbar_arrive_expect_tx(bar(kCeBarFull + s), (uint32_t)kCeStageBytes);
                        tma_load_2d(sbase + s * kCeStageBytes, &tm_h, bar(kCeBarFull + s), ks * kCeK, rt * kCeM);
                        tma_load_2d(sbase + s * kCeStageBytes + kCeABytes, &tm_w, bar(kCeBarFull + s), ks * kCeK,
                                    vb * kCeN);
                    }
                    __syncwarp();
                }
            }
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------------ MMA issuer
        const uint32_t idesc = make_idesc_bf16(kCeM, kCeN, 0);
        uint32_t it = 0, blk = 0;
        bool ok = true;
#pragma unroll 1
        for (int tl = 0; tl < n_units && ok; ++tl) {
            const int u = (int)blockIdx.x + tl * (int)gridDim.x;
            int pn, rt;
            ce_unit(p, u, pn, rt);
            const int vb_end = min(p.nvb, (pn + 1) * p.panel);
#pragma unroll 1
            for (int vb = pn * p.panel; vb < vb_end && ok; ++vb, ++blk) {
                const uint32_t a = blk & 1u;
                // the accumulator half is free once the fold warps have read block blk - 2 out of it
                ok = mbar_wait_warp(bar(kCeBarAccFree + a), ((blk >> 1) & 1) ^ 1, abort_flag, p.status, kErrCeMma);
                if (!ok) break;
                tc_fence_after();
#pragma unroll 1
                for (int ks = 0; ks < p.ksteps; ++ks, ++it) {
                    const uint32_t s = it % kCeStages;
                    ok = mbar_wait_warp(bar(kCeBarFull + s), (it / kCeStages) & 1, abort_flag, p.status, kErrCeMma);
                    if (!ok) break;
                    tc_fence_after();
                    const uint64_t a_desc = make_smem_desc(sbase + s * kCeStageBytes, 0, 1024);
                    const uint64_t b_desc = make_smem_desc(sbase + s * kCeStageBytes + kCeABytes, 0, 1024);
                    if (elect_one_sync()) {
#pragma unroll
                        for (int kk = 0; kk < kCeK / 16; ++kk)
                            mma_ss(tmem + a * kCeN, a_desc + (uint64_t)((kk * 32) >> 4), b_desc + (uint64_t)((kk * 32) >> 4),
                                   idesc, (ks > 0 || kk > 0) ? 1u : 0u);
                        tc_commit(bar(kCeBarEmpty + s));
                        if (ks == p.ksteps - 1) tc_commit(bar(kCeBarAccFull + a));
                    }
                    __syncwarp();
                }
            }
        }
    } else if (warp >= 4) {
        // ------------------------------------------------------------------ fold warps (4..7)
        const int q4 = warp & 3;
        const int row = 32 * q4 + lane;
        const uint32_t lane_addr = (uint32_t)(32 * q4) << 16;
        uint32_t blk = 0;
        bool ok = true;
#pragma unroll 1
        for (int tl = 0; tl < n_units && ok; ++tl) {
            const int u = (int)blockIdx.x + tl * (int)gridDim.x;
            int pn, rt;
            ce_unit(p, u, pn, rt);
            const int vb_end = min(p.nvb, (pn + 1) * p.panel);
            const int grow = rt * kCeM + row;
            const bool valid = grow < p.R;
            const int z = valid ? p.target[grow] : -1;
            float m = -INFINITY, l = 0.f, zt = 0.f;  // running max and sum in the log2 domain
            bool have_zt = false;
#pragma unroll 1
            for (int vb = pn * p.panel; vb < vb_end && ok; ++vb, ++blk) {
                const uint32_t a = blk & 1u;
                ok = mbar_wait_warp(bar(kCeBarAccFull + a), (blk >> 1) & 1, abort_flag, p.status, kErrCeFold);
                if (!ok) break;
                tc_fence_after();
                const int col0 = vb * kCeN;
                const int ncol = min(kCeN, p.V - col0);  // real vocabulary entries in this block
#pragma unroll 1
                for (int c = 0; c < kCeN / 32; ++c) {
                    if (c * 32 >= ncol) break;  // warp-uniform: nothing real in the remaining chunks
                    uint32_t rr[32];
                    tmem_ld32(tmem + lane_addr + a * kCeN + c * 32, rr);
                    tmem_wait_ld();
                    const int zrel = z - col0 - c * 32;
                    if (__any_sync(0xffffffffu, (unsigned)zrel < 32u)) {
#pragma unroll
                        for (int i = 0; i < 32; ++i)
                            if (zrel == i) { zt = __uint_as_float(rr[i]); have_zt = true; }
                    }
                    float y[32];
                    float cmax = -INFINITY;
                    const int nreal = ncol - c * 32;  // >= 1
#pragma unroll
                    for (int i = 0; i < 32; ++i) {
                        y[i] = i < nreal ? __uint_as_float(rr[i]) * kLog2e : -INFINITY;
                        cmax = fmaxf(cmax, y[i]);
                    }
                    if (cmax > m) {
                        l *= ex2_approx(m - cmax);  // 2^-inf = 0 on the first chunk
                        m = cmax;
                    }
                    float s0 = 0.f, s1 = 0.f;
#pragma unroll
                    for (int i = 0; i < 32; i += 2) {
                        s0 += ex2_approx(y[i] - m);
                        s1 += ex2_approx(y[i + 1] - m);
                    }
                    l += s0 + s1;
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(bar(kCeBarAccFree + a));
            }
            if (ok && valid) {
                p.part[(size_t)grow * p.npanel + pn] = make_float2(m, l);
                if (have_zt) p.tlogit[grow] = zt;
            }
        }
    }

    if (*abort_flag != 0) __nanosleep(20000);
    tc_fence_before();
    __syncthreads();
    if (warp == 2) tmem_dealloc(tmem, 512);
}

// Merges the partials of a row (contiguous, one lane each) into lse and nll by one warp, and forms the masked average of a
// candidate.  WHOLE: a block per candidate does both, its warps taking the rows in turn.  Else a block takes kCeFinalWarps rows
// of the list of all rows, and ce_average_kernel follows.  (One thread per row, walking over the panels, took 13 to 30 us in
// calls whose projection takes 40 to 400.)
constexpr int kCeFinalWarps = 8;
// Up to three rows per warp a second launch costs more than it gives.  Whole calls, one kernel and two: 1 candidate x 8 rows
// (Dm = 1024, 32 000 words) 18.2 and 19.6 us, x 20 21.0 and 20.5, x 32 20.4 and 18.6, x 64 21.7 and 15.5, x 256 52 and 21; 512 x
// 20 (Dm = 256, 4 096 words) 37.9 and 38.2, x 96 144 and 139; 1 x 30 000 (Dm = 256, 4 096 words) 3 660 and 98.
constexpr int kCeWholeRows = 24;
template <bool WHOLE>
__global__ void __launch_bounds__(32 * kCeFinalWarps)
ce_finalize_kernel(const float2 *part, const float *tlogit, const int *target, const float *mask, float *nll, float *lse,
                   float *loss, long long R, int Lr, int npanel, int V)
{
    __shared__ float num_s[kCeFinalWarps], den_s[kCeFinalWarps];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    float num = 0.f, den = 0.f;
    const long long first = (long long)blockIdx.x * (WHOLE ? Lr : kCeFinalWarps), end = WHOLE ? first + Lr : min(R, first + kCeFinalWarps);
    for (long long r = first + warp; r < end; r += kCeFinalWarps) {
        const float2 *pr = part + (size_t)r * npanel;
        float M = -INFINITY, L = 0.f;
        for (int pn = lane; pn < npanel; pn += 32) {
            const float2 x = pr[pn];
            const float m = fmaxf(M, x.x);
            // (equal maxima need no factor; a lane that has seen no panel holds -inf, and -inf - -inf is not 0)
            L = (M == m ? L : L * exp2f(M - m)) + (x.x == m ? x.y : x.y * exp2f(x.x - m));
            M = m;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const float m2 = __shfl_xor_sync(0xffffffffu, M, o), l2 = __shfl_xor_sync(0xffffffffu, L, o);
            const float m = fmaxf(M, m2);
            L = (M == m ? L : L * exp2f(M - m)) + (m2 == m ? l2 : l2 * exp2f(m2 - m));
            M = m;
        }
        const float ls = (M + log2f(L)) * kLn2;
        const float w = mask[r];
        float v = 0.f;
        if (w != 0.f) {
            const int z = target[r];
            v = (z >= 0 && z < V) ? w * (ls - tlogit[r]) : __int_as_float(0x7fc00000);  // a bad token id shows as NaN
        }
        if (lane == 0) {
            lse[r] = ls;
            nll[r] = v;
        }
        num += v;
        den += w;
    }
    if (!WHOLE) return;
    if (lane == 0) {
        num_s[warp] = num;
        den_s[warp] = den;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        num = den = 0.f;
        for (int k = 0; k < kCeFinalWarps; ++k) {
            num += num_s[k];
            den += den_s[k];
        }
        loss[blockIdx.x] = den != 0.f ? num / den : 0.f;
    }
}

// Masked average of a candidate of many rows: one block per candidate.
__global__ void __launch_bounds__(32 * kCeFinalWarps)
ce_average_kernel(const float *nll, const float *mask, float *loss, int Lr)
{
    __shared__ float num_s[kCeFinalWarps], den_s[kCeFinalWarps];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    float num = 0.f, den = 0.f;
    for (int i = threadIdx.x; i < Lr; i += 32 * kCeFinalWarps) {
        const size_t r = (size_t)blockIdx.x * Lr + i;
        num += nll[r];
        den += mask[r];
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        num += __shfl_xor_sync(0xffffffffu, num, o);
        den += __shfl_xor_sync(0xffffffffu, den, o);
    }
    if (lane == 0) {
        num_s[warp] = num;
        den_s[warp] = den;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        num = den = 0.f;
        for (int k = 0; k < kCeFinalWarps; ++k) {
            num += num_s[k];
            den += den_s[k];
        }
        loss[blockIdx.x] = den != 0.f ? num / den : 0.f;
    }
}

inline bool encode_2d(CUtensorMap *map, const void *base, int cols, long long rows, int box_rows)
{
    cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
    cuuint64_t str[1] = {(cuuint64_t)cols * 2};
    cuuint32_t box[2] = {64, (cuuint32_t)box_rows};
    return encode_map(map, base, 2, dims, str, box);
}

struct CePlan {
    int nrt, nvb, panel, npanel, Rpad, ksteps;
    size_t ws_bytes;
};

// Units a call may have: the workspace holds the partials of that many.  It never falls as rows are added, so that scratch
// sized for a program's largest batch serves its smaller ones, and depends on the sizes alone, so that the query gives the same
// bytes wherever it is made.  32 units for each of 148 SMs, or panels of five blocks, leave out no width that
// would be more than half a percent cheaper.
long long ce_max_units(int nrt, int nvb)
{
    const long long narrow = (long long)nvb * nrt, cap = 32 * 148, wide = (long long)((nvb + 4) / 5) * nrt;
    return wide > cap ? wide : narrow < cap ? narrow : cap;
}

// Blocks per panel: a CTA's time is its units times their blocks, so the width is the one whose units fill the last
// round of the SMs best, 8 where nothing is clearly better.  204 rows of a 32 000-word vocabulary are 32 units of
// 8 blocks on 148 SMs, or 250 of one; 10 240 rows of 128 256 words 34.05 rounds of 8, or 38.9 of 7.  Whole calls at
// Dm = 4096 against 8 blocks throughout: 204 rows x 32 000 words 191 -> 77 us, 270 x 128 256 449 -> 366, 512 x 32 000
// 193 -> 130, 3 540 x 32 000 815 -> 711, 10 240 x 128 256 8.10 -> 7.98 ms.
int ce_panel(int nrt, int nvb)
{
    const int sms = sm_count();
    const long long most = ce_max_units(nrt, nvb);
    auto cost = [&](int panel) {
        const long long units = (long long)((nvb + panel - 1) / panel) * nrt;
        return (double)((units + sms - 1) / sms) * (panel + 0.1);
    };
    int best = 8;
    double best_cost = 0.99 * cost(8);
    for (int panel = kCeMaxPanel; panel >= 1; --panel)
        if (cost(panel) < best_cost && (long long)((nvb + panel - 1) / panel) * nrt <= most) {
            best = panel;
            best_cost = cost(panel);
        }
    return best;
}

CePlan ce_plan(long long R, int Dm, int V)
{
    CePlan pl;
    pl.nrt = (int)((R + kCeM - 1) / kCeM);
    pl.nvb = (V + kCeN - 1) / kCeN;
    pl.panel = ce_panel(pl.nrt, pl.nvb);
    pl.npanel = (pl.nvb + pl.panel - 1) / pl.panel;
    pl.Rpad = pl.nrt * kCeM;
    pl.ksteps = (Dm + kCeK - 1) / kCeK;
    pl.ws_bytes = (size_t)ce_max_units(pl.nrt, pl.nvb) * kCeM * sizeof(float2) + (size_t)pl.Rpad * sizeof(float);
    return pl;
}

}  // namespace

bool ce_fwd_supported(int N, int Lr, int Dm, int V)
{
    if (N < 1 || Lr < 1 || Dm < 8 || V < 1 || Dm % 8 != 0) return false;  // row pitch must be a multiple of 16 bytes
    const long long R = (long long)N * Lr;
    if (R > 16000000ll || (long long)V > 4000000ll) return false;
    const CePlan pl = ce_plan(R, Dm, V);
    return (long long)pl.npanel * pl.nrt < 2000000000ll;
}

size_t ce_fwd_workspace_bytes(int N, int Lr, int Dm, int V)
{
    return ce_plan((long long)N * Lr, Dm, V).ws_bytes;
}

cudaError_t launch_ce_fwd(const CeArgs &a, void *workspace, unsigned int *status_word, cudaStream_t stream)
{
    const long long R = (long long)a.N * a.Lr;
    const CePlan pl = ce_plan(R, a.Dm, a.V);
    CUtensorMap tm_h, tm_w;
    if (!encode_2d(&tm_h, a.hidden, a.Dm, R, kCeM)) return cudaErrorInvalidValue;
    if (!encode_2d(&tm_w, a.weight, a.Dm, a.V, kCeN)) return cudaErrorInvalidValue;
    CeParams p;
    p.target = a.target;
    p.part = static_cast<float2 *>(workspace);
    p.tlogit = reinterpret_cast<float *>(p.part + (size_t)pl.npanel * pl.Rpad);
    p.status = status_word;
    p.R = (int)R; p.Dm = a.Dm; p.V = a.V;
    p.nrt = pl.nrt; p.nvb = pl.nvb; p.panel = pl.panel; p.npanel = pl.npanel; p.units = pl.npanel * pl.nrt; p.ksteps = pl.ksteps;
    p.rg = sm_count() / 4 < 1 ? 1 : sm_count() / 4;
    if (p.rg > pl.nrt) p.rg = pl.nrt;
    const int smem_bytes = kCeStages * kCeStageBytes + 8 * kCeNumBars + 64;
    static PerDeviceOnce attr_set;
    if (cudaError_t e = ensure_max_smem(ce_fwd_kernel, attr_set, smem_bytes); e != cudaSuccess) return e;
    const int grid = p.units < sm_count() ? p.units : sm_count();
    {
        KernelTiming timing(kKernelCeFwd, stream);
        ce_fwd_kernel<<<grid, kCeThreads, smem_bytes, stream>>>(tm_h, tm_w, p);
    }
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    {
        KernelTiming timing(kKernelCeFinalize, stream);
        const bool whole = a.Lr <= kCeWholeRows;
        const unsigned blocks = whole ? (unsigned)a.N : (unsigned)((R + kCeFinalWarps - 1) / kCeFinalWarps);
        auto kernel = whole ? ce_finalize_kernel<true> : ce_finalize_kernel<false>;
        kernel<<<blocks, 32 * kCeFinalWarps, 0, stream>>>(p.part, p.tlogit, a.target, a.mask, a.nll, a.lse, a.loss, R, a.Lr,
                                                          pl.npanel, a.V);
        if (!whole) ce_average_kernel<<<(unsigned)a.N, 32 * kCeFinalWarps, 0, stream>>>(a.nll, a.mask, a.loss, a.Lr);
        count_launches(whole ? 2 : 3);
    }
    return cudaGetLastError();
}

}  // namespace pskv
