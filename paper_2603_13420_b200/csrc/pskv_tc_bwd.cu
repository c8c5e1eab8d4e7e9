// Shared-prefix attention backward for sm_100a (tcgen05 / TMEM / TMA), one kernel for all three gradients:
//   dQ        = scale * sum_j dS_j K_j              over the shared prefix keys and the visible suffix keys
//   dK_suffix = scale * sum over rows of dS^T Q     (suffix keys only: the prefix cache is frozen, Sec. 4.2)
//   dV_suffix =         sum over rows of  P^T dO
//   with P = exp(S - lse), S = scale Q K^T, dP = dO V^T, dS = P o (dP - D), D = <dO, O> (a pre-pass, or in here: DSource).
// Q and dO are fetched once; nothing is read or recomputed twice except in the passes named below.
//
// A CTA works on units.  A unit is `cu` neighbouring candidates of one KV head, so that the sums over rows
// and heads that make dK_suffix / dV_suffix stay inside the CTA: its rows (n_rep * S per candidate, padded
// to Rp, a multiple of 8) are cut into 128-row tiles.  A tile meets its keys in pieces of 64: the pieces of
// the prefix, and for every candidate it touches the pieces of that candidate's suffix (several short
// candidates share a piece).  One (tile, piece) pair is an item:
//   S  = Q K^T, dP = dO V^T       (M = 128 rows, N = keys)   -> one of two tensor-memory slots
//   dS (and for suffix pieces P)  element-wise, bf16, to shared memory
//   dQ += dS K                    (M = 128 rows, N = d)
//   suffix pieces: dV^T += dO^T P, dK^T += Q^T dS   (M = d, N = keys, K = rows)
// The second and third products read the very tiles the first ones read, as operands of the other major-ness.
//
// What bounds it: HBM for head layouts with one query head per KV head (every row's q, dout, k, v and three
// gradients move once), else the chain of an item.  64 keys instead of 128 per item cost a third more shared
// memory reads by the tensor cores (768 instead of 512 cycles for a 128 x 128 score block and its dP), but two
// S/dP slots fit beside dQ and the accumulators, and because dS goes to shared memory a slot is handed back
// as soon as the element-wise warps have loaded it, before their arithmetic: the next scores never wait
// for the previous item's dQ.
//
// Measured (whole forward + backward step, before: a dQ kernel and a suffix-gradient kernel that each read q and
// dout, for S a multiple of 8 and up to 64, CUDA-core kernels for the rest): B = 512, 32/8 heads, P = 256, S = 48
// 563 -> 519 us; B = 128, 32/32 heads, P = 160, S = 40 171 -> 142 us; B = 100, 32/32 heads, P = 78, S = 113 10.4 ms ->
// 0.30 ms (0.32 with two terms, below).  With a staging buffer for dQ instead of four K and three V stages (three and two fit): 529 us.
//
// Suffixes beyond 64 keys have several pieces per candidate but only one pair of accumulators (128 columns).
// When the unit is one tile the pieces take turns; when it is several tiles, pass 0 accumulates piece 0 (and
// all of dQ) and every later pass walks over the tiles once more for one further piece.
//
// Launches of few candidates (the gradient of a search's one current suffix) are split: every tile's dQ and every
// suffix piece's dK / dV is a unit of its own, so that one candidate keeps up to tiles + pieces SMs per KV head
// busy instead of one, at the price of forming the scores of the suffix pieces once more.  Whole steps: B = 1, 32/8
// heads, P = 78, S = 113 45 -> 25 us; B = 4, 32/8, P = 1000, S = 100 96 -> 56; B = 20, 32/8, P = 200, S = 90 84 -> 77 (with
// one term; with two 28, 59 and 80).
//
// Two terms (TWO): P and dS go to shared memory as sums of two bf16 values (16 bits of mantissa), and the contractions run over
// both.  Taken where the suffix length is no multiple of 8 or exceeds 64 (multiples of 8 up to 128: for dK / dV alone):
// the CUDA-core kernels, which these lengths came from, hold P and dS in fp32, and one bf16 term is not that.  Distance
// (2-norm) of dQ / dK / dV from 64-bit gradients, B = 333, 32/8 heads, P = 217, S = 53: CUDA cores 2.40e-3 / 1.80e-3 / 1.67e-3,
// one term 3.25e-3 / 2.51e-3 / 2.35e-3, two terms 2.40e-3 / 1.80e-3 / 1.67e-3 (the rounding of the results, and of `out` inside
// D).  Price of the second term, kernel and pre-pass: that shape 290 -> 312 us, B = 100, 32/32 heads, P = 78, S = 113 192 ->
// 223, B = 250, 32/8, P = 385, S = 42 210 -> 256, one candidate, 32/8, P = 78, S = 113 17.2 -> 19.9 (CUDA cores: 21.4 ms, 10.3 ms,
// 20 ms, 233 us).  The second terms take the memory of three stages; with three K stages and one V stage left the
// second and third of these took 243 and 271 us, with two and two 266 and 310 (both with the spills the loop had then).
//
// Persistent CTA, one per SM, 24 warps:
//   warp 0      TMA producer: K and V pieces (two rings); writes the descriptor of every item
//   warp 1      tcgen05.mma issuer: S and dP
//   warp 2      tcgen05.mma issuer: dQ, dV^T, dK^T (owns the TMEM allocation)
//   warp 3      TMA producer: Q and dO tiles; writes the row table of every tile
//   warps 4-19  element-wise: two sets of eight warps take the items in turn; a warp covers 32 rows x 32 keys
//   warps 20-23 epilogue: dQ, dK and dV from tensor memory to global memory
// The walk over units, tiles and pieces is done by the producers (and the epilogue); the MMA issuers and the
// element-wise warps follow 16-byte descriptors in shared memory.  With the walk in every role the registers it
// took spilled and the roles' loops ran 900 to 2 900 cycles an item of bookkeeping.
// Every wait is bounded.
#include <string.h>

#include "pskv_common.cuh"
#include "pskv_sm100.cuh"
#include "pskv_tc_common.cuh"

namespace pskv {
namespace {

using namespace sm100;

constexpr int kPieceN = 64;   // keys per item
constexpr int kThreads = 32 * 24;
constexpr int kMaxRing = 4;
constexpr int kMaxInstr = kMaxFusedInstructions;  // prefixes one launch can serve
// tensor memory: two (S, dP) slots, dQ, the two transposed accumulators
constexpr int kSlotCols = 128, kColDp = 64, kColDq = 256, kColDv = 384, kColDk = 448;
constexpr int kDsBytes = kTileM * 128;  // P or dS of an item: 128 rows x 64 keys of bf16

enum : unsigned int {
    kErrProdKv = 0x201, kErrProdQ = 0x202, kErrMmaS = 0x203, kErrMmaGrad = 0x204, kErrElem = 0x205,
    kErrEpi = 0x206, kErrAlign = 0x207
};

struct TcBwdParams {
    const float *lse;      // [B*Hq*S] from the forward pass
    const float *row_dot;  // [B*Hq*S] D, or (kDWarps) what it is formed from:
    const __nv_bfloat16 *out, *dout;
    const float *dlse;     // gradient on lse, or nullptr
    __nv_bfloat16 *dq;       // [B,Hq,S,d]
    __nv_bfloat16 *dk, *dv;  // [B,Hkv,S,d]
    unsigned int *status;
    float sl2;             // scale * log2(e)
    float scale;
    int dq_sectors;        // dq is 32-byte aligned
    int dq_two;            // TWO: dQ over both terms too
    int Hq, Hkv, S, P, n_rep;
    int Rg;                // rows of a candidate in one KV-head group: n_rep * S
    int Rp;                // rows it takes in the unit's row list: Rg rounded up to 8
    int Sp;                // key columns a candidate takes in a piece that holds several: S rounded up to 8
    int cu;                // candidates per unit
    int cpp;               // candidates per suffix piece (> 1 only when a unit is one tile)
    int nh;                // suffix pieces per candidate: ceil(S / 64)
    int seg, cbox;         // rows and candidates of one Q / dO box
    int sfx_box;           // key rows per candidate in a suffix K / V box
    int nblk;              // prefix pieces: ceil(P / 64)
    int Kq;                // candidates per instruction (all of them when there is one prefix)
    int upi, upg;          // units per (KV head, instruction), per KV head
    int n_units;
    int n_tiles, n_sub;    // split launch: dQ units and all units of a candidate (else n_sub = 1)
    FastDiv fd_upg, fd_upi, fd_sub, fd_Rp, fd_S, fd_cpp;
    int stages_k, stages_v;
    int off_do, off_q, off_k, off_v, off_p, off_ds, off_rows, off_bar, off_misc;
    int zero_lo, zero_hi;  // operand buffers with rows that no copy may reach before the MMAs read them
    int pad[kMaxInstr];    // left padding of each instruction's prefix cache (Sec. 4.3)
};

// Where the row statistic D comes from: a pre-pass over dout and out; the element-wise warps, plain FMAs under the first copies
// (every CTA has one tile); an item of its own in front of a tile's others, whose scores are dO O^T.
enum DSource { kDTable = 0, kDWarps = 1, kDItem = 2 };

template <int D>
struct Cfg {
    static constexpr int kSlabs = D / 64;              // 64-column (128-byte) swizzle slabs per row
    static constexpr int kSlabBytes = kTileM * 128;    // slab of a 128-row tile
    static constexpr int kTileBytes = kSlabs * kSlabBytes;
    static constexpr int kPieceSlab = kPieceN * 128;   // slab of a 64-row K / V piece
    static constexpr int kPieceBytes = kSlabs * kPieceSlab;
};

enum {
    kBarQFull = 0,   // Q of a tile landed (kJoint: and dO)
    kBarDoFull,      // dO of a tile landed
    kBarQFree,       // the last MMA of each issuer that reads them has completed (2 arrivals)
    kBarDqFull,      // dQ of a tile is final
    kBarDqFree,      // the epilogue has read it out (4 arrivals)
    kBarPFree,       // the MMAs that read P have completed
    kBarAccFull,     // the accumulators are final
    kBarAccFree,     // the epilogue has read them out (4 arrivals)
    kBarSFull,                       // [2] S and dP of an item are in tensor memory
    kBarSFree = kBarSFull + 2,       // [2] the element-wise warps have loaded them (8 arrivals)
    kBarDsReady = kBarSFree + 2,     // [2] dS (and P) of an item are in shared memory (8 arrivals)
    kBarDsFree = kBarDsReady + 2,    // [2] the MMAs that read dS have completed
    kBarRowsFull = kBarDsFree + 2,   // [2] the row table of a tile is written
    kBarDFull = kBarRowsFull + 2,    // [2] kDItem: D is in the row table (8 arrivals)
    kBarKFull = kBarDFull + 2,       // (also: the item's descriptor is written)
    kBarVFull = kBarKFull + kMaxRing,
    kBarKFree = kBarVFull + kMaxRing,
    kBarVFree = kBarKFree + kMaxRing,
    kNumBars = kBarVFree + kMaxRing
};
constexpr int kBarBytes = 512;
constexpr int kDescOff = 384;   // descriptors behind the barriers: eight entries of 16 bytes
static_assert(kNumBars * 8 <= kDescOff && kDescOff + 8 * 16 <= kBarBytes, "barrier area");
constexpr int kRowsBytes = 2 * kTileM * 8;  // row tables (-lse log2(e), D) of two tiles

// Descriptor of an item.  x: MMA N and the flags below; y: suffix item: candidate group, prefix item: first and
// last real key (8 bits each); z: first key of the piece inside the suffix; w: running number of the tile.
// At most five items are between the producer (which needs a free K stage) and the element-wise warps, so
// eight entries are enough.
enum : uint32_t {
    kDescN = 0x7f, kDescSfx = 1u << 7, kDescAcc = 1u << 8, kDescAccFirst = 1u << 9, kDescAccLast = 1u << 10,
    kDescQDone = 1u << 11,     // last item of the tile that feeds dK / dV: its products are the last to read Q and dO
    kDescLast = 1u << 12, kDescDq = 1u << 13, kDescFirst = 1u << 14,
    kDescAccOdd = 1u << 15,    // parity of the items that fed dK / dV so far
    kDescK0 = 16, kDescK1 = 20,  // rows of the group inside the tile, in steps of 16 (4 bits each)
    kDescRowDot = 1u << 24,      // the item of the tile's row statistic (x holds nothing else)
    kDescEnd = 1u << 31
};

// The walk over units, passes and tiles, the same in every role.  SPLIT: the units are the parts of a candidate (an
// instantiation of its own: with the decision at run time the other launches were 4 % slower).
template <bool SPLIT>
struct Walk {
    int u, u_end;           // unit
    int g, inst, b0, ncand; // its KV head, instruction, first candidate, candidates
    int t_first, t_end, npass, pass, tt;
    bool dq_;               // SPLIT: see dq(), fed()
    int fed_;
    int R0, rows;           // tile: first row of the unit's row list, rows that belong to the unit
    int grp_lo, ngrp;       // candidate groups (pieces' worth of candidates) the tile touches
    int kp0;                // first prefix piece (pieces of padding only are left out)
    int n_sfx, n_items;     // suffix items, all items of the tile

    __device__ __forceinline__ bool done() const { return u >= u_end; }
    // the pass forms dQ (and walks over the prefix)
    __device__ __forceinline__ bool dq() const { return SPLIT ? dq_ : pass == 0; }
    // pieces that feed dK / dV: 0 none, 1 all, 2 the one of number `pass`
    __device__ __forceinline__ int fed() const { return SPLIT ? fed_ : npass > 1 ? 2 : 1; }

    __device__ __forceinline__ void unit(const TcBwdParams &p)
    {
        if (done()) return;
        const int w = SPLIT ? p.fd_sub.div(u) : u;
        g = p.fd_upg.div(w);
        const int r = w - g * p.upg;
        inst = p.fd_upi.div(r);
        const int ub = r - inst * p.upi;
        b0 = inst * p.Kq + ub * p.cu;
        ncand = min(p.cu, p.Kq - ub * p.cu);
        kp0 = p.pad[inst] / kPieceN;
        t_first = pass = 0;
        t_end = (ncand * p.Rp + kTileM - 1) / kTileM;
        npass = t_end > 1 ? p.nh : 1;
        if (SPLIT) {
            const int sub = u - w * p.n_sub;
            if (sub < p.n_tiles) {
                t_first = sub;
                t_end = sub + 1;
                npass = 1;
                dq_ = true;
                fed_ = 0;
            } else {
                pass = sub - p.n_tiles;
                npass = pass + 1;
                dq_ = false;
                fed_ = 2;
            }
        }
        tt = t_first;
        tile(p);
    }
    __device__ __forceinline__ void tile(const TcBwdParams &p)
    {
        R0 = tt * kTileM;
        rows = min(kTileM, ncand * p.Rp - R0);
        grp_lo = p.fd_cpp.div(p.fd_Rp.div(R0));
        ngrp = p.fd_cpp.div(p.fd_Rp.div(R0 + rows - 1)) - grp_lo + 1;
        n_sfx = dq() ? ngrp * p.nh : ngrp;
        n_items = n_sfx + (dq() ? p.nblk - kp0 : 0);
    }
    __device__ __forceinline__ void start(const TcBwdParams &p)
    {
        u = (int)((long long)blockIdx.x * p.n_units / gridDim.x);
        u_end = (int)((long long)(blockIdx.x + 1) * p.n_units / gridDim.x);
        unit(p);
    }
    __device__ __forceinline__ void next_tile(const TcBwdParams &p)
    {
        if (++tt < t_end) { tile(p); return; }
        if (++pass < npass) {
            tt = t_first;
            tile(p);
            return;
        }
        ++u;
        unit(p);
    }
    // suffix item j of the tile: candidate group and 64-key piece of its suffix
    __device__ __forceinline__ int grp(const TcBwdParams &p, int j) const
    {
        return grp_lo + (!dq() || p.nh == 1 ? j : j / p.nh);
    }
    __device__ __forceinline__ int half(const TcBwdParams &p, int j) const
    {
        return !dq() ? pass : p.nh == 1 ? 0 : j - j / p.nh * p.nh;
    }
    __device__ __forceinline__ bool acc(int h) const { return fed() == 1 || (fed() == 2 && h == pass); }  // feeds dK / dV
    __device__ __forceinline__ int grp_row0(const TcBwdParams &p, int gr) const { return gr * p.cpp * p.Rp; }
    __device__ __forceinline__ int grp_row1(const TcBwdParams &p, int gr) const
    {
        return min((gr + 1) * p.cpp, ncand) * p.Rp;
    }
    // key columns of a suffix item
    __device__ __forceinline__ int sfx_cols(const TcBwdParams &p, int gr, int h) const
    {
        if (p.nh > 1) return min(kPieceN, p.S - h * kPieceN);
        return p.cpp == 1 ? p.S : min(p.cpp, ncand - gr * p.cpp) * p.Sp;
    }
};

// 32 bytes of a row, a whole sector in one instruction where the alignment allows it.  dQ goes to memory this way,
// straight from the epilogue's registers: lane <-> row, so an instruction covers 32 full sectors of 32 rows.  (With
// 16-byte stores, half a sector each, such a store is slow; a staging buffer and TMA stores need 32 KB that
// the K / V rings use better.)
__device__ __forceinline__ void store_sector(__nv_bfloat16 *dst, const uint32_t *v, bool aligned)
{
    if (aligned) {
        asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(dst), "r"(v[0]), "r"(v[1]), "r"(v[2]),
                     "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7])
                     : "memory");
    } else {
        reinterpret_cast<uint4 *>(dst)[0] = make_uint4(v[0], v[1], v[2], v[3]);
        reinterpret_cast<uint4 *>(dst)[1] = make_uint4(v[4], v[5], v[6], v[7]);
    }
}

// Eight values as bf16; `two`: with what the rounding leaves (exact in fp32) as bf16 in the buffer behind.
__device__ __forceinline__ void store_terms(uint32_t dst, const float *x, bool two)
{
    uint32_t hi[4], lo[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) hi[i] = pack_bf16x2(x[2 * i], x[2 * i + 1]);
    st_shared_v4(dst, hi);
    if (!two) return;
#pragma unroll
    for (int i = 0; i < 4; ++i)
        lo[i] = pack_bf16x2(x[2 * i] - __uint_as_float(hi[i] << 16), x[2 * i + 1] - __uint_as_float(hi[i] & 0xffff0000u));
    st_shared_v4(dst + kDsBytes, lo);
}

// The rows [first, first + 8) of a CTA's one tile: (-lse log2(e), D) into the row table, D = <dout, out> less the
// gradient on lse, formed as the pre-pass does.
template <int D>
__device__ __forceinline__ void row_dots(const TcBwdParams &p, int b0, int g, int R0, int rows, float2 *table, int first, int lane)
{
    constexpr int kLanes = D / 8, kRows = 32 / kLanes, kLoads = 8 / kRows;  // lanes of a row, rows of a load
    const int sub = lane / kLanes, col = lane % kLanes * 8;
    uint4 o[kLoads], d[kLoads];
    float2 st[kLoads];
#pragma unroll
    for (int u = 0; u < kLoads; ++u) {
        const int row = first + u * kRows + sub, R = R0 + row, c = p.fd_Rp.div(R), r = R - c * p.Rp;
        const bool v = row < rows && r < p.Rg;  // rows that do not exist get probability zero
        o[u] = d[u] = make_uint4(0, 0, 0, 0);
        st[u] = make_float2(-INFINITY, 0.f);
        if (v) {
            const size_t at = ((size_t)(b0 + c) * p.Hq + (size_t)g * p.n_rep) * p.S + r;
            o[u] = *reinterpret_cast<const uint4 *>(p.out + at * D + col);
            d[u] = *reinterpret_cast<const uint4 *>(p.dout + at * D + col);
            st[u] = make_float2(-p.lse[at] * kLog2e, p.dlse ? p.dlse[at] : 0.f);
        }
    }
#pragma unroll
    for (int u = 0; u < kLoads; ++u) {
        const __nv_bfloat162 *ob = reinterpret_cast<const __nv_bfloat162 *>(&o[u]);
        const __nv_bfloat162 *gb = reinterpret_cast<const __nv_bfloat162 *>(&d[u]);
        float acc = 0.f;
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const float2 x = __bfloat1622float2(ob[e]), y = __bfloat1622float2(gb[e]);
            acc = fmaf(x.x, y.x, acc);
            acc = fmaf(x.y, y.y, acc);
        }
#pragma unroll
        for (int off = kLanes / 2; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
        if (lane % kLanes == 0)
            table[first + u * kRows + sub] = make_float2(st[u].x, acc - st[u].y);
    }
}

// DSRC: where D comes from (DSource).  TWO: P and dS as two terms.
template <int D, bool SPLIT, int DSRC, bool TWO>
__global__ void __launch_bounds__(kThreads, 1)
tc_bwd_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_do,
              const __grid_constant__ CUtensorMap tm_pk, const __grid_constant__ CUtensorMap tm_pv,
              const __grid_constant__ CUtensorMap tm_sk, const __grid_constant__ CUtensorMap tm_sv,
              const __grid_constant__ CUtensorMap tm_out, const __grid_constant__ TcBwdParams p)
{
    using C = Cfg<D>;
    constexpr bool DROW = DSRC == kDWarps, DOT = DSRC == kDItem;
    constexpr int kTerms = TWO ? 2 : 1;
    constexpr bool kEight = TWO || DOT;
    // Q and dO on one barrier: launches with few items to a tile, or with one tile to a CTA (see the S / dP issuer).
    constexpr bool kJoint = SPLIT || DROW;
    constexpr uint64_t kLoTerm = (uint64_t)(kDsBytes >> 4);  // descriptor distance from a P / dS buffer to its second term
    extern __shared__ __align__(1024) uint8_t smem[];
    const int tid = threadIdx.x, lane = tid & 31;
    const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
    PSKV_TRACE_DECL;
    grid_dep_launch();  // the next kernel of the stream may take over SMs as this one's CTAs exit
    const uint32_t sbase = smem_u32(smem);
    const uint32_t bar0 = sbase + p.off_bar;
    auto bar = [&](int i) { return bar0 + 8u * (uint32_t)i; };
    volatile int *abort_flag = reinterpret_cast<volatile int *>(smem + p.off_misc + 4);
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(smem + p.off_misc);

    if ((sbase & 1023u) != 0u) {  // the swizzled layouts need a 1024-byte aligned base
        if (tid == 0) atomicCAS(p.status, 0u, (unsigned int)kErrAlign);
        return;
    }
    // Operand rows that no copy ever writes must hold finite values (0 * NaN would poison a sum).  Zeroing all
    // buffers in every launch, with the barriers set up by one thread, cost 2 us: one candidate, 32/8 heads, P = 78, S =
    // 113 22.9 instead of 20.9 us, 12 candidates, 32/32 heads, P = 90, S = 77 27.0 instead of 24.9.
    for (int i = p.zero_lo / 16 + tid; i < p.zero_hi / 16; i += kThreads)
        reinterpret_cast<uint4 *>(smem)[i] = make_uint4(0, 0, 0, 0);
    if (warp == 3) {
#pragma unroll 1
        for (int i = lane; i < kNumBars; i += 32) {
            const bool epi = i == kBarDqFree || i == kBarAccFree;
            const bool elem = (i >= kBarSFree && i < kBarSFree + 2) || (i >= kBarDsReady && i < kBarDsReady + 2);
            mbar_init(bar(i), elem || (i >= kBarDFull && i < kBarDFull + 2) ? 8u : epi ? 4u : i == kBarQFree ? 2u : DROW && i == kBarRowsFull ? 16u : 1u);
        }
        if (lane == 0) *abort_flag = 0;
        fence_barrier_init();
    }
    fence_proxy_async();
    if (warp == 2) {
        tmem_alloc(smem_u32(tmem_slot), 512);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    // everything above touched shared and tensor memory only: it may run under the tail of the kernel before
    grid_dep_wait();

    Walk<SPLIT> w;
    w.start(p);
    bool ok = true;

    if (warp == 0) {
        // ------------------------------------------------------------------ producer: K and V pieces
        if (lane == 0) {
            prefetch_tensormap(&tm_sk);
            prefetch_tensormap(&tm_sv);
            if (p.P > 0) { prefetch_tensormap(&tm_pk); prefetch_tensormap(&tm_pv); }
        }
        int ks = 0, vs = 0;
        uint32_t kph = 1, vph = 1, item = 0, tile = 0, n_acc = 0;
        const uint32_t sfx_tx = (uint32_t)(C::kSlabs * p.sfx_box * p.cpp * 128);
        uint4 *descs = reinterpret_cast<uint4 *>(smem + p.off_bar + kDescOff);
#pragma unroll 1
        for (; !w.done() && ok; w.next_tile(p), ++tile) {
            const int head = w.inst * p.Hkv + w.g;
            if (DOT) {
                // the item of the row statistic: rows of `out`, columns 0-63 into a K stage, 64-127 into a V stage
                const int step = p.seg * p.cbox, nb = (w.rows + step - 1) / step;
                const int R = w.R0 + lane * step, c = p.fd_Rp.div(R), r = R - c * p.Rp;
                ok = mbar_wait_warp(bar(kBarKFree + ks), kph, abort_flag, p.status, kErrProdKv);
                if (ok) ok = mbar_wait_warp(bar(kBarVFree + vs), vph, abort_flag, p.status, kErrProdKv);
                if (!ok) break;
                const uint32_t kb = bar(kBarKFull + ks), vb = bar(kBarVFull + vs);
                if (lane == 0) {
                    descs[item & 7u] = make_uint4(kDescRowDot, 0u, 0u, (tile & 0xffffu) | (uint32_t)w.tt << 16);
                    mbar_arrive_expect_tx(kb, (uint32_t)(nb * step * 128));
                    mbar_arrive_expect_tx(vb, (uint32_t)(nb * step * 128));
                }
                __syncwarp();
                if (lane < nb) {
                    const uint32_t off = (uint32_t)(lane * step * 128);
                    tma_load_4d(sbase + p.off_k + ks * C::kPieceBytes + off, &tm_out, kb, 0, r, w.g, w.b0 + c);
                    tma_load_4d(sbase + p.off_v + vs * C::kPieceBytes + off, &tm_out, vb, 64, r, w.g, w.b0 + c);
                }
                __syncwarp();
                if (++ks == p.stages_k) { ks = 0; kph ^= 1u; }
                if (++vs == p.stages_v) { vs = 0; vph ^= 1u; }
                ++item;
            }
            // suffix items are spread evenly over the tile's items, the first one first: their accumulators are drained, and
            // their P buffer is read, under the prefix items in between
            int e = 0, j = 0, q = 0;
            bool sfx = true;
#pragma unroll 1
            for (int k = 0; k < w.n_items; ++k, ++item) {
                int row, b = w.b0, n;
                uint4 dsc;
                dsc.x = (k == w.n_items - 1 ? kDescLast : 0u) | (k == 0 ? kDescFirst : 0u) | (w.dq() ? kDescDq : 0u) |
                        (w.fed() == 0 && k == w.n_items - 1 ? kDescQDone : 0u);
                dsc.w = (tile & 0xffffu) | (uint32_t)w.tt << 16;
                if (sfx) {
                    const int h = w.half(p, j), gr = w.grp(p, j);
                    row = h * kPieceN;
                    b += gr * p.cpp;
                    n = w.sfx_cols(p, gr, h);
                    dsc.x |= kDescSfx;
                    dsc.y = (uint32_t)gr;
                    dsc.z = (uint32_t)row;
                    if (w.acc(h)) {
                        const int r0 = w.grp_row0(p, gr) - w.R0, r1 = w.grp_row1(p, gr) - w.R0;
                        dsc.x |= kDescAcc | (r0 >= 0 ? kDescAccFirst : 0u) | (r1 <= kTileM ? kDescAccLast : 0u) |
                                 ((n_acc & 1u) ? kDescAccOdd : 0u) | (uint32_t)(max(r0, 0) >> 4) << kDescK0 |
                                 (uint32_t)((min(r1, kTileM) + 15) >> 4) << kDescK1;
                        if (gr == w.grp_lo + w.ngrp - 1 && (w.fed() == 2 || h == p.nh - 1)) dsc.x |= kDescQDone;
                        ++n_acc;
                    }
                } else {
                    row = (w.kp0 + q) * kPieceN;
                    n = min(kPieceN, p.P - row);
                    dsc.y = (uint32_t)max(0, p.pad[w.inst] - row) | (uint32_t)(n - 1) << 8;
                    dsc.z = 0u;
                }
                dsc.x |= (uint32_t)((n + 15) & ~15);
                const uint32_t tx = sfx ? sfx_tx : (uint32_t)C::kPieceBytes;
                ok = mbar_wait_warp(bar(kBarKFree + ks), kph, abort_flag, p.status, kErrProdKv);
                if (!ok) break;
                if (elect_one_sync()) {
                    descs[item & 7u] = dsc;
                    const uint32_t dst = sbase + p.off_k + ks * C::kPieceBytes, fb = bar(kBarKFull + ks);
                    mbar_arrive_expect_tx(fb, tx);
#pragma unroll
                    for (int sl = 0; sl < C::kSlabs; ++sl) {
                        if (sfx) tma_load_4d(dst + sl * C::kPieceSlab, &tm_sk, fb, sl * 64, row, w.g, b);
                        else tma_load_3d(dst + sl * C::kPieceSlab, &tm_pk, fb, sl * 64, row, head);
                    }
                }
                __syncwarp();
                ok = mbar_wait_warp(bar(kBarVFree + vs), vph, abort_flag, p.status, kErrProdKv);
                if (!ok) break;
                if (elect_one_sync()) {
                    const uint32_t dst = sbase + p.off_v + vs * C::kPieceBytes, fb = bar(kBarVFull + vs);
                    mbar_arrive_expect_tx(fb, tx);
#pragma unroll
                    for (int sl = 0; sl < C::kSlabs; ++sl) {
                        if (sfx) tma_load_4d(dst + sl * C::kPieceSlab, &tm_sv, fb, sl * 64, row, w.g, b);
                        else tma_load_3d(dst + sl * C::kPieceSlab, &tm_pv, fb, sl * 64, row, head);
                    }
                }
                __syncwarp();
                if (++ks == p.stages_k) { ks = 0; kph ^= 1u; }
                if (++vs == p.stages_v) { vs = 0; vph ^= 1u; }
                if (sfx) ++j; else ++q;
                e += w.n_sfx;
                if (e >= w.n_items) e -= w.n_items;
                sfx = e < w.n_sfx;
            }
        }
        // two end marks, one for each set of element-wise warps
#pragma unroll 1
        for (int i = 0; i < 2 && ok; ++i, ++item) {
            ok = mbar_wait_warp(bar(kBarKFree + ks), kph, abort_flag, p.status, kErrProdKv);
            if (ok && elect_one_sync()) {
                descs[item & 7u] = make_uint4(kDescEnd, 0u, 0u, 0u);
                mbar_arrive(bar(kBarKFull + ks));
            }
            __syncwarp();
            if (++ks == p.stages_k) { ks = 0; kph ^= 1u; }
        }
    } else if (warp == 3) {
        // ------------------------------------------------------------------ producer: Q and dO tiles
        if (lane == 0) {
            prefetch_tensormap(&tm_q);
            prefetch_tensormap(&tm_do);
        }
        const int step = p.seg * p.cbox;  // rows of one box
        uint32_t tile = 0;
#pragma unroll 1
        while (!w.done() && ok) {
            // The tile's row table: -lse log2(e) and D; rows that do not exist get probability zero.
            float st[4], dr[4];
#pragma unroll
            for (int i = 0; i < 4 && !DROW; ++i) {
                const int row = 32 * i + lane, R = w.R0 + row;
                const int c = p.fd_Rp.div(R), r = R - c * p.Rp;
                const bool v = row < w.rows && r < p.Rg;
                const size_t at = ((size_t)(w.b0 + c) * p.Hq + (size_t)w.g * p.n_rep) * p.S + r;
                st[i] = v ? -p.lse[at] * kLog2e : -INFINITY;
                dr[i] = v && !DOT ? p.row_dot[at] : 0.f;
            }
            const int nb = (w.rows + step - 1) / step;
            const int R = w.R0 + lane * step;
            const int c = p.fd_Rp.div(R), r = R - c * p.Rp, g = w.g, b = w.b0 + c;
            // While idle, ask for the next tile's rows in L2: the buffers are single, so their copies can only
            // be issued right when they are needed.
            w.next_tile(p);
            if (!w.done() && lane < (w.rows + step - 1) / step) {
                const int Rn = w.R0 + lane * step;
                const int cn = p.fd_Rp.div(Rn), rn = Rn - cn * p.Rp;
#pragma unroll
                for (int sl = 0; sl < C::kSlabs; ++sl) {
                    tma_prefetch_4d(&tm_q, sl * 64, rn, w.g, w.b0 + cn);
                    tma_prefetch_4d(&tm_do, sl * 64, rn, w.g, w.b0 + cn);
                }
            }
            __syncwarp();
            ok = mbar_wait_warp(bar(kBarQFree), (tile & 1u) ^ 1u, abort_flag, p.status, kErrProdQ);
            if (!ok) break;
            PSKV_TRACE_EVENT(2, tile);
            const uint32_t tx = (uint32_t)(nb * C::kSlabs * step * 128);
            if (lane == 0) {
                if (!kJoint) mbar_arrive_expect_tx(bar(kBarDoFull), tx);
                mbar_arrive_expect_tx(bar(kBarQFull), kJoint ? 2 * tx : tx);
            }
            __syncwarp();
            if (lane < nb) {
#pragma unroll
                for (int sl = 0; sl < C::kSlabs; ++sl) {
                    const uint32_t off = (uint32_t)(sl * C::kSlabBytes + lane * step * 128);
                    tma_load_4d(sbase + p.off_do + off, &tm_do, bar(kJoint ? kBarQFull : kBarDoFull), sl * 64, r, g, b);
                }
#pragma unroll
                for (int sl = 0; sl < C::kSlabs; ++sl) {
                    const uint32_t off = (uint32_t)(sl * C::kSlabBytes + lane * step * 128);
                    tma_load_4d(sbase + p.off_q + off, &tm_q, bar(kBarQFull), sl * 64, r, g, b);
                }
            }
            if (!DROW) {
                // Table tile & 1 was last read for tile - 2; the MMAs behind kBarQFree of tile - 1 came after that.
                float2 *rows = reinterpret_cast<float2 *>(smem + p.off_rows) + (tile & 1u) * kTileM;
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    if (DOT) rows[32 * i + lane].x = st[i];  // (the element-wise warps add D)
                    else rows[32 * i + lane] = make_float2(st[i], dr[i]);
                }
                __syncwarp();
                if (lane == 0) mbar_arrive(bar(kBarRowsFull + (tile & 1u)));
            }
            ++tile;
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------------ S = Q K^T, dP = dO V^T
        const uint64_t q_desc = make_smem_desc(sbase + p.off_q, 0, 1024);
        const uint64_t do_desc = make_smem_desc(sbase + p.off_do, 0, 1024);
        const uint4 *descs = reinterpret_cast<const uint4 *>(smem + p.off_bar + kDescOff);
        int ks = 0, vs = 0;
        uint32_t kph = 0, vph = 0;
#pragma unroll 1
        for (uint32_t item = 0;; ++item) {
            const uint32_t slot = item & 1u;
            const uint32_t d_tmem = tmem + slot * kSlotCols;
            const uint64_t k_desc = make_smem_desc(sbase + p.off_k + ks * C::kPieceBytes, 0, 1024);
            const uint64_t v_desc = make_smem_desc(sbase + p.off_v + vs * C::kPieceBytes, 0, 1024);
            PSKV_TRACE_EVENT(12, item);
            ok = mbar_wait_warp(bar(kBarKFull + ks), kph, abort_flag, p.status, kErrMmaS);
            if (!ok) break;
            const uint32_t x = __shfl_sync(0xffffffffu, descs[item & 7u].x, 0);
            if (x & kDescEnd) break;
            const uint32_t idesc = make_idesc_bf16(kTileM, (int)(x & kDescN), 0);
            const uint32_t tile_ph = descs[item & 7u].w & 1u;
            if (x & (DOT ? kDescRowDot : kDescFirst)) ok = mbar_wait_warp(bar(kJoint ? kBarQFull : kBarDoFull), tile_ph, abort_flag, p.status, kErrMmaS);
            if (ok) ok = mbar_wait_warp(bar(kBarSFree + slot), ((item >> 1) & 1u) ^ 1u, abort_flag, p.status, kErrMmaS);
            if (ok) ok = mbar_wait_warp(bar(kBarVFull + vs), vph, abort_flag, p.status, kErrMmaS);
            if (!ok) break;
            PSKV_TRACE_EVENT(15, item);
            tc_fence_after();
            // dP first: its V piece is handed back while S is under way (with two terms there is one V stage, and its next piece
            // is what the following item waits for), and a tile's first dP starts when dO has landed, before Q.  Whole steps:
            // 58 candidates, 32/32 heads, P = 1735, S = 66 601 -> 569 us, 61, 32/32, P = 1206, S = 54 314 -> 303, 14, 32/32, P = 417, S =
            // 123 97 -> 94; in one term no change.  (Split launches have few items to a tile, and where a CTA has one tile nothing runs
            // before it; waiting for the two in turn costs them more: one candidate, 32/8, P = 78, S = 113 27.9 -> 28.8; the
            // backward of 64, 4/4, d = 64, P = 256, S = 40 12.70 -> 12.86, of 40 12.18 -> 12.35.)
            if (DOT && (x & kDescRowDot)) {
                // dO O^T over the whole slot: 64 columns of O from the K stage, 64 from the V stage
                if (elect_one_sync()) {
                    constexpr uint32_t idesc_dot = make_idesc_bf16(kTileM, kTileM, 0);
#pragma unroll 1
                    for (uint32_t i = 0; i < D / 32; ++i) mma_ss(d_tmem, do_desc + 2 * i, k_desc + 2 * i, idesc_dot, i);
#pragma unroll 1
                    for (uint32_t i = 0; i < D / 32; ++i)
                        mma_ss(d_tmem, do_desc + (C::kSlabBytes >> 4) + 2 * i, v_desc + 2 * i, idesc_dot, 1u);
                    tc_commit(bar(kBarSFull + slot));
                    tc_commit(bar(kBarVFree + vs));
                }
                __syncwarp();
                if (++ks == p.stages_k) { ks = 0; kph ^= 1u; }
                if (++vs == p.stages_v) { vs = 0; vph ^= 1u; }
                continue;
            }
            if (elect_one_sync()) {
#pragma unroll
                for (int i = 0; i < D / 16; ++i) {
                    const uint64_t aoff = (uint64_t)(((i >> 2) * C::kSlabBytes + (i & 3) * 32) >> 4);
                    const uint64_t boff = (uint64_t)(((i >> 2) * C::kPieceSlab + (i & 3) * 32) >> 4);
                    mma_ss(d_tmem + kColDp, do_desc + aoff, v_desc + boff, idesc, i > 0 ? 1u : 0u);
                }
                tc_commit(bar(kBarVFree + vs));
            }
            if (!kJoint && (x & kDescFirst)) {
                __syncwarp();
                ok = mbar_wait_warp(bar(kBarQFull), tile_ph, abort_flag, p.status, kErrMmaS);
                if (!ok) break;
                tc_fence_after();
            }
            if (elect_one_sync()) {
#pragma unroll
                for (int i = 0; i < D / 16; ++i) {
                    const uint64_t aoff = (uint64_t)(((i >> 2) * C::kSlabBytes + (i & 3) * 32) >> 4);
                    const uint64_t boff = (uint64_t)(((i >> 2) * C::kPieceSlab + (i & 3) * 32) >> 4);
                    mma_ss(d_tmem, q_desc + aoff, k_desc + boff, idesc, i > 0 ? 1u : 0u);
                }
                tc_commit(bar(kBarSFull + slot));
                if (x & kDescLast) tc_commit(bar(kBarQFree));
            }
            __syncwarp();
            PSKV_TRACE_EVENT(10, item);
            if (++ks == p.stages_k) { ks = 0; kph ^= 1u; }
            if (++vs == p.stages_v) { vs = 0; vph ^= 1u; }
        }
    } else if (warp == 2) {
        // ------------------------------------------------------------------ dQ += dS K, dV^T += dO^T P, dK^T += Q^T dS
        const uint32_t idesc_dq = make_idesc_bf16(kTileM, D, 1);
        // A operands with d contiguous.  Head dim 128: two 64-column slabs of dO / of Q.  Head dim 64: M is still
        // 128, rows 0-63 from the slab of dO and rows 64-127 from the slab of Q, which lies behind it.
        const uint64_t dot_desc = make_smem_desc(sbase + p.off_do, D == 128 ? C::kSlabBytes : p.off_q - p.off_do, 1024);
        const uint64_t qt_desc = D == 128 ? make_smem_desc(sbase + p.off_q, C::kSlabBytes, 1024) : dot_desc;
        const uint64_t p_desc = make_smem_desc(sbase + p.off_p, kDsBytes, 1024);
        const uint4 *descs = reinterpret_cast<const uint4 *>(smem + p.off_bar + kDescOff);
        int ks = 0;
        uint32_t kph = 0, dqph = 1, accph = 1;
#pragma unroll 1
        for (uint32_t item = 0;; ++item) {
            const uint32_t slot = item & 1u;
            const uint64_t ds_a = make_smem_desc(sbase + p.off_ds + slot * kTerms * kDsBytes, kDsBytes, 1024);
            const uint64_t k_desc = make_smem_desc(sbase + p.off_k + ks * C::kPieceBytes, C::kPieceSlab, 1024);
            ok = mbar_wait_warp(bar(kBarKFull + ks), kph, abort_flag, p.status, kErrMmaGrad);
            if (!ok) break;
            const uint32_t x = __shfl_sync(0xffffffffu, descs[item & 7u].x, 0);
            if (x & kDescEnd) break;
            const int n = (int)(x & kDescN);
            const uint32_t acc0 = (x & kDescFirst) ? 0u : 1u;
            PSKV_TRACE_EVENT(13, item);
            ok = mbar_wait_warp(bar(kBarDsReady + slot), (item >> 1) & 1u, abort_flag, p.status, kErrMmaGrad);
            if (ok && (x & (kDescDq | kDescFirst)) == (kDescDq | kDescFirst)) {  // the previous dQ must have been read out
                ok = mbar_wait_warp(bar(kBarDqFree), dqph, abort_flag, p.status, kErrMmaGrad);
                dqph ^= 1u;
            }
            if (!ok) break;
            tc_fence_after();
            if ((x & kDescDq) && elect_one_sync()) {
#pragma unroll
                for (int i = 0; i < kPieceN / 16; ++i)
                    if (i * 16 < n)
                        mma_ss(tmem + kColDq, ds_a + (uint64_t)(i * 32 >> 4), k_desc + (uint64_t)(i * 2048 >> 4), idesc_dq,
                               i > 0 ? 1u : acc0);
                if (TWO && p.dq_two) {
#pragma unroll
                    for (int i = 0; i < kPieceN / 16; ++i)
                        if (i * 16 < n)
                            mma_ss(tmem + kColDq, ds_a + kLoTerm + (uint64_t)(i * 32 >> 4), k_desc + (uint64_t)(i * 2048 >> 4), idesc_dq, 1u);
                }
            }
            __syncwarp();
            if (x & kDescAcc) {
                if (x & kDescAccFirst) {
                    PSKV_TRACE_EVENT(16, item);
                    ok = mbar_wait_warp(bar(kBarAccFree), accph, abort_flag, p.status, kErrMmaGrad);
                    accph ^= 1u;
                    if (!ok) break;
                    tc_fence_after();
                }
                PSKV_TRACE_EVENT(11, item);
                const uint32_t idesc_acc = make_idesc_bf16_ab(128, n, 1, 1);
                // rows of the tile that belong to the group, in steps of 16 (the others among them are zero in P and dS, for finite inputs)
                const int k0 = (int)((x >> kDescK0) & 15u), k1 = (int)((x >> kDescK1) & 15u);
                if (elect_one_sync()) {
                    uint32_t a = (x & kDescAccFirst) ? 0u : 1u;
#pragma unroll 1
                    for (int i = k0; i < k1; ++i) {
                        const uint64_t off = (uint64_t)(i * (2048 >> 4));
                        mma_ss(tmem + kColDv, dot_desc + off, p_desc + off, idesc_acc, a);
                        mma_ss(tmem + kColDk, qt_desc + off, ds_a + off, idesc_acc, a);
                        a = 1u;
                        if (TWO) {
                            mma_ss(tmem + kColDv, dot_desc + off, p_desc + kLoTerm + off, idesc_acc, 1u);
                            mma_ss(tmem + kColDk, qt_desc + off, ds_a + kLoTerm + off, idesc_acc, 1u);
                        }
                    }
                    tc_commit(bar(kBarPFree));
                    if (x & kDescAccLast) tc_commit(bar(kBarAccFull));
                }
                __syncwarp();
            }
            if (elect_one_sync()) {
                if (x & kDescQDone) tc_commit(bar(kBarQFree));
                tc_commit(bar(kBarDsFree + slot));
                tc_commit(bar(kBarKFree + ks));
                if ((x & (kDescLast | kDescDq)) == (kDescLast | kDescDq)) tc_commit(bar(kBarDqFull));
            }
            __syncwarp();
            PSKV_TRACE_EVENT(14, item);
            if (++ks == p.stages_k) { ks = 0; kph ^= 1u; }
        }
    } else if (warp < 20) {
        // ------------------------------------------------------------------ element-wise warps (4..19)
        const int set = (warp - 4) >> 3;        // items of parity `set`
        const int c0 = ((warp >> 2) & 1) ? 0 : 32;   // my 32 of the piece's 64 keys
        const int row = 32 * (warp & 3) + lane;
        const uint32_t my_tmem = tmem + ((uint32_t)(32 * (warp & 3)) << 16) + set * kSlotCols + c0;
        // (32-bit addresses: the loop has no registers to spare)
        const uint32_t p_row = sbase + p.off_p + row * 128;
        const uint32_t ds_row = sbase + p.off_ds + set * kTerms * kDsBytes + row * 128;
        const uint32_t descs = bar0 + kDescOff, rows_at = sbase + p.off_rows + row * 8;
        int ks = set;
        uint32_t kph = 0, tile = 0xffffffffu;  // (no tile has this number and index)
        if (ks >= p.stages_k) { ks -= p.stages_k; kph ^= 1u; }
        if (DROW) {  // under the first copies
            row_dots<D>(p, w.b0, w.g, w.R0, w.rows, reinterpret_cast<float2 *>(smem + p.off_rows),
                        32 * (warp & 3) + 8 * ((warp - 4) >> 2), lane);
            __syncwarp();
            if (lane == 0) mbar_arrive(bar(kBarRowsFull));
        }
        float neg_lse2 = 0.f, drow = 0.f;
        int my_grp = -1, my_lo = 0, my_hi = 0;
#pragma unroll 1
        for (uint32_t item = (uint32_t)set;; item += 2) {
            const uint32_t sph = (item >> 1) & 1u;
            PSKV_TRACE_EVENT(26, item);
            ok = mbar_wait_warp(bar(kBarKFull + ks), kph, abort_flag, p.status, kErrElem);
            if (!ok) break;
            const uint4 dsc = ld_shared_v4(descs + (item & 7u) * 16);
            if (dsc.x & kDescEnd) break;
            ks += 2;
            if (ks >= p.stages_k) {
                ks -= p.stages_k;
                kph ^= 1u;
            }
            if (DOT && (dsc.x & kDescRowDot)) {
                // Rows 32 q .. 32 q + 31 have their diagonal in columns 32 q .. 32 q + 31 of the slot; my sixteen of them are
                // those of lanes c0 / 2 .. c0 / 2 + 15.  Rows that do not exist (-lse is -infinity) get 0.
                ok = mbar_wait_warp(bar(kBarSFull + set), sph, abort_flag, p.status, kErrElem);
                if (!ok) break;
                tc_fence_after();
                uint32_t rs[16];
                tmem_ld16(my_tmem - c0 + 32 * (warp & 3) + (c0 >> 1), rs);
                tmem_wait_ld();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(bar(kBarSFree + set));
#pragma unroll
                for (int h = 8; h > 0; h >>= 1)
#pragma unroll
                    for (int i = 0; i < h; ++i) rs[i] = (lane & h) ? rs[i + h] : rs[i];
                ok = mbar_wait_warp(bar(kBarRowsFull + (dsc.w & 1u)), (dsc.w >> 1) & 1u, abort_flag, p.status, kErrElem);
                if (!ok) break;
                if ((lane & 16) == (c0 >> 1)) {
                    const uint32_t at = rows_at + (dsc.w & 1u) * (kTileM * 8);
                    st_shared_f(at + 4, ld_shared_f(at) == -INFINITY ? 0.f : __uint_as_float(rs[0]));
                }
                __syncwarp();
                if (lane == 0) mbar_arrive(bar(kBarDFull + (dsc.w & 1u)));
                // (nothing was written to dS, but its barriers go on item by item)
                ok = mbar_wait_warp(bar(kBarDsFree + set), sph ^ 1u, abort_flag, p.status, kErrElem);
                if (!ok) break;
                if (lane == 0) mbar_arrive(bar(kBarDsReady + set));
                continue;
            }
            if (dsc.w != tile) {
                tile = dsc.w;
                ok = mbar_wait_warp(bar((DOT ? kBarDFull : kBarRowsFull) + (tile & 1u)), (tile >> 1) & 1u, abort_flag, p.status, kErrElem);
                if (!ok) break;
                const float2 rt = ld_shared_f2(rows_at + (tile & 1u) * (kTileM * 8));
                neg_lse2 = rt.x;
                drow = rt.y;
                // candidate group of my row, first key column of its candidate in the piece, last visible one
                const int R = (int)(tile >> 16) * kTileM + row, c = p.fd_Rp.div(R), r = R - c * p.Rp;
                my_grp = p.fd_cpp.div(c);
                my_lo = (c - my_grp * p.cpp) * p.Sp;
                my_hi = my_lo + r - p.fd_S.div(r) * p.S;
            }
            const bool acc = (dsc.x & kDescAcc) != 0u;
            int lo, hi;  // visible columns of my row
            if (dsc.x & kDescSfx) {
                const bool mine = (int)dsc.y == my_grp;
                lo = mine ? my_lo : 1;
                hi = mine ? my_hi - (int)dsc.z : 0;
            } else {
                lo = (int)(dsc.y & 0xffu);
                hi = (int)(dsc.y >> 8);
            }
            // my 32 columns: 0 = not read by the MMAs, 1 = nothing visible to any row of this warp (zeros),
            // 2 = some masked, 3 = all visible to all rows
            int kind = 0;
            if (c0 < (int)(dsc.x & kDescN)) {
                const bool all_valid = lo <= c0 && hi >= c0 + 31;
                const bool none_valid = hi < lo || hi < c0 || lo > c0 + 31;
                kind = __all_sync(0xffffffffu, all_valid) ? 3 : __all_sync(0xffffffffu, none_valid) ? 1 : 2;
            }
            PSKV_TRACE_EVENT(25, item);
            ok = mbar_wait_warp(bar(kBarSFull + set), sph, abort_flag, p.status, kErrElem);
            if (!ok) break;
            PSKV_TRACE_EVENT(20, item);
            tc_fence_after();
#pragma unroll
            for (int hf = 0; hf < 2; ++hf) {
                uint32_t rs[16], rd[16], pk[8], pp[8];
                if (kind >= 2) {
                    tmem_ld16(my_tmem + hf * 16, rs);
                    tmem_ld16(my_tmem + kColDp + hf * 16, rd);
                    tmem_wait_ld();
                }
                if (hf == 1) {
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(bar(kBarSFree + set));
                }
                if (kEight) {
                    // eight columns at a time, stored as they are made (the waits first): with sixteen of P and dS held in
                    // fp32 across the waits the loop spilled
                    if (hf == 0) {
                        PSKV_TRACE_EVENT(21, item);
                        ok = mbar_wait_warp(bar(kBarDsFree + set), sph ^ 1u, abort_flag, p.status, kErrElem);
                        if (ok && acc)
                            ok = mbar_wait_warp(bar(kBarPFree), (dsc.x & kDescAccOdd) ? 0u : 1u, abort_flag, p.status, kErrElem);
                        if (!ok) break;
                        PSKV_TRACE_EVENT(22, item);
                    }
                    if (kind == 0) continue;
                    const bool lo_term = TWO && (acc || p.dq_two);
#pragma unroll
                    for (int i = 0; i < 2; ++i) {
                        float e[8], ds[8];
                        if (kind >= 2) {
#pragma unroll
                            for (int c = 0; c < 8; c += 2) {
                                float x0 = __uint_as_float(rs[8 * i + c]), x1 = __uint_as_float(rs[8 * i + c + 1]);
                                fma_f32x2(x0, x1, p.sl2, neg_lse2);
                                e[c] = ex2_approx(x0);
                                e[c + 1] = ex2_approx(x1);
                            }
                            if (kind == 2) {
                                const unsigned span = (unsigned)(hi - lo);
                                const int base = c0 + hf * 16 + 8 * i - lo;
                                const bool any_col = hi >= lo;
#pragma unroll
                                for (int c = 0; c < 8; ++c) e[c] = (any_col && (unsigned)(base + c) <= span) ? e[c] : 0.f;
                            }
#pragma unroll
                            for (int c = 0; c < 8; c += 2) {
                                ds[c] = __uint_as_float(rd[8 * i + c]);
                                ds[c + 1] = __uint_as_float(rd[8 * i + c + 1]);
                                add_f32x2(ds[c], ds[c + 1], -drow, -drow);
                                mul_f32x2(ds[c], ds[c + 1], e[c], e[c + 1]);
                            }
                        } else {
#pragma unroll
                            for (int c = 0; c < 8; ++c) e[c] = ds[c] = 0.f;
                        }
                        const int off = (((c0 >> 3) + 2 * hf + i) ^ (row & 7)) << 4;
                        store_terms(ds_row + off, ds, lo_term);
                        if (acc) store_terms(p_row + off, e, TWO);
                    }
                    continue;
                }
                if (kind >= 2) {
                    float e[16];
#pragma unroll
                    for (int i = 0; i < 16; i += 2) {
                        float x0 = __uint_as_float(rs[i]), x1 = __uint_as_float(rs[i + 1]);
                        fma_f32x2(x0, x1, p.sl2, neg_lse2);
                        e[i] = ex2_approx(x0);
                        e[i + 1] = ex2_approx(x1);
                    }
                    if (kind == 2) {
                        const unsigned span = (unsigned)(hi - lo);
                        const int base = c0 + hf * 16 - lo;
                        const bool any_col = hi >= lo;
#pragma unroll
                        for (int i = 0; i < 16; ++i) e[i] = (any_col && (unsigned)(base + i) <= span) ? e[i] : 0.f;
                    }
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        float d0 = __uint_as_float(rd[2 * i]), d1 = __uint_as_float(rd[2 * i + 1]);
                        add_f32x2(d0, d1, -drow, -drow);
                        mul_f32x2(d0, d1, e[2 * i], e[2 * i + 1]);
                        pk[i] = pack_bf16x2(d0, d1);
                        pp[i] = pack_bf16x2(e[2 * i], e[2 * i + 1]);
                    }
                } else {
#pragma unroll
                    for (int i = 0; i < 8; ++i) pk[i] = pp[i] = 0u;
                }
                if (hf == 0) {
                    PSKV_TRACE_EVENT(21, item);
                    ok = mbar_wait_warp(bar(kBarDsFree + set), sph ^ 1u, abort_flag, p.status, kErrElem);
                    if (ok && acc)
                        ok = mbar_wait_warp(bar(kBarPFree), (dsc.x & kDescAccOdd) ? 0u : 1u, abort_flag, p.status, kErrElem);
                    if (!ok) break;
                    PSKV_TRACE_EVENT(22, item);
                }
                if (kind != 0) {
                    // 128-byte rows, 16-byte chunks swizzled by the row
#pragma unroll
                    for (int i = 0; i < 2; ++i) {
                        const int off = (((c0 >> 3) + 2 * hf + i) ^ (row & 7)) << 4;
                        st_shared_v4(ds_row + off, pk + 4 * i);
                        if (acc) st_shared_v4(p_row + off, pp + 4 * i);
                    }
                }
            }
            if (!ok) break;
            fence_proxy_async();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar(kBarDsReady + set));
            PSKV_TRACE_EVENT(24, item);
        }
    } else {
        // ------------------------------------------------------------------ epilogue warps (20..23)
        const int ew = warp & 3;
        const int row = 32 * ew + lane;
        const uint32_t lane_addr = (uint32_t)(32 * ew) << 16;
        uint32_t dqph = 0, accph = 0;
#pragma unroll 1
        for (; !w.done() && ok; w.next_tile(p)) {
#pragma unroll 1
            for (int j = 0; j < w.n_sfx; ++j) {
                const int h = w.half(p, j), gr = w.grp(p, j);
                if (!w.acc(h) || w.grp_row1(p, gr) > w.R0 + kTileM) continue;
                // ---- accumulators of a candidate group: lane <-> column d, tensor-memory column <-> key
                ok = mbar_wait_warp(bar(kBarAccFull), accph, abort_flag, p.status, kErrEpi);
                if (!ok) break;
                accph ^= 1u;
                PSKV_TRACE_EVENT(30, w.u);
                tc_fence_after();
                const int n = w.sfx_cols(p, gr, h);
                int b = w.b0 + gr * p.cpp, t = h * kPieceN;   // candidate and key of the coming eight columns
                const int b_end = w.b0 + w.ncand;
#pragma unroll 1
                for (int col = 0; col < n; col += 16) {
                    uint32_t av[16], ak[16];
                    if (D == 128 || ew < 2) tmem_ld16(tmem + lane_addr + kColDv + col, av);
                    if (D == 128 || ew >= 2) tmem_ld16(tmem + lane_addr + kColDk + col, ak);
                    tmem_wait_ld();
                    if (col + 16 >= n) {
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(bar(kBarAccFree));
                    }
#pragma unroll
                    for (int i8 = 0; i8 < 16; i8 += 8) {
                        // eight columns lie inside one candidate (Sp is a multiple of 8)
                        const size_t o = (((size_t)b * p.Hkv + w.g) * p.S + t) * D + (D == 128 ? row : row & 63);
                        const int nk = b < b_end ? p.S - t : 0;
                        if (D == 128 || ew < 2) {
                            __nv_bfloat16 *dst = p.dv + o;
#pragma unroll
                            for (int i = 0; i < 8; ++i)
                                if (i < nk) dst[i * D] = __float2bfloat16_rn(__uint_as_float(av[i8 + i]));
                        }
                        if (D == 128 || ew >= 2) {
                            __nv_bfloat16 *dst = p.dk + o;
#pragma unroll
                            for (int i = 0; i < 8; ++i)
                                if (i < nk) dst[i * D] = __float2bfloat16_rn(__uint_as_float(ak[i8 + i]) * p.scale);
                        }
                        t += 8;
                        if (t == p.Sp && p.cpp > 1) {
                            t = 0;
                            ++b;
                        }
                    }
                }
                PSKV_TRACE_EVENT(31, w.u);
            }
            if (!ok) break;
            if (!w.dq()) continue;
            // ---- dQ of the tile
            ok = mbar_wait_warp(bar(kBarDqFull), dqph, abort_flag, p.status, kErrEpi);
            if (!ok) break;
            dqph ^= 1u;
            PSKV_TRACE_EVENT(33, w.u);
            tc_fence_after();
            const int R = w.R0 + row, c = p.fd_Rp.div(R), r = R - c * p.Rp;
            const bool stored = row < w.rows && r < p.Rg;
            __nv_bfloat16 *dst = p.dq + (((size_t)(w.b0 + c) * p.Hq + (size_t)w.g * p.n_rep) * p.S + r) * D;
#pragma unroll 1
            for (int q4 = 0; q4 < D / 32; ++q4) {
                uint32_t o[32], v[16];
                tmem_ld32(tmem + lane_addr + kColDq + q4 * 32, o);
                tmem_wait_ld();
                if (q4 == D / 32 - 1) {
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(bar(kBarDqFree));
                }
#pragma unroll
                for (int i = 0; i < 16; ++i)
                    v[i] = pack_bf16x2(__uint_as_float(o[2 * i]) * p.scale, __uint_as_float(o[2 * i + 1]) * p.scale);
                if (stored) {
                    store_sector(dst + q4 * 32, v, p.dq_sectors != 0);
                    store_sector(dst + q4 * 32 + 16, v + 8, p.dq_sectors != 0);
                }
            }
            PSKV_TRACE_EVENT(34, w.u);
        }
    }

    PSKV_TRACE_FLUSH;
    if (*abort_flag != 0) __nanosleep(20000);  // let copies and MMAs still in flight drain
    tc_fence_before();
    __syncthreads();
    if (warp == 2) tmem_dealloc(tmem, 512);
}

// ------------------------------------------------------------------------------ host side

struct BwdPlan {
    bool ok;
    int cu, cpp, nh, Rp, Sp, seg, cbox, sfx_box, nblk, upi;
    int n_tiles, n_sub;
    int terms;             // bf16 terms of P and dS
    int stages_k, stages_v;
    int off_do, off_q, off_k, off_v, off_p, off_ds, off_rows, off_bar, off_misc, smem_bytes;
};

// Chooses the candidates per unit and lays out shared memory.  The cost of a choice is what the busiest SM
// does: its units times their items (64-key pieces summed over tiles and passes) plus a fixed share per tile,
// worth about one item.
BwdPlan make_plan(const Dims &dm, int n_instr)
{
    BwdPlan pl;
    memset(&pl, 0, sizeof(pl));
    const int Rg = dm.n_rep * dm.S, Kq = dm.B / n_instr;
    pl.Sp = round_up(dm.S, 8);
    pl.nh = (dm.S + kPieceN - 1) / kPieceN;
    pl.nblk = (dm.P + kPieceN - 1) / kPieceN;
    const int sms = sm_count();
    double best = -1.0;
    // A candidate's rows may be padded further than to the next multiple of 8: 4 heads x 42 rows are two tiles, one of
    // them a third full, or, as 176 rows, three tiles for two candidates (kernel alone, one term, B = 250, P = 385 240 -> 203 us;
    // 4 x 67 rows, B = 100, P = 300 181 -> 169; 4 x 35, B = 144, P = 92 74 -> 66).
    for (int Rp = round_up(Rg, 8); Rp < Rg + 64; Rp += 8) {
        const int seg = gcd_int(Rp, kTileM);
        for (int cu = 1; cu <= 16 && cu <= Kq; ++cu) {
            const int tiles = (cu * Rp + kTileM - 1) / kTileM;
            // a tile that straddles candidates takes 128 / seg boxes
            if (cu > 1 && ((tiles > 1 && seg < 16) || tiles > 12)) break;
            int cpp = 1, sfx = 0;
            if (tiles == 1) {
                cpp = pl.nh > 1 ? 1 : kPieceN / pl.Sp < cu ? kPieceN / pl.Sp : cu;
                sfx = (cu + cpp - 1) / cpp * pl.nh;
            } else {
                for (int t = 0; t < tiles; ++t) {
                    const int r1 = (t + 1) * kTileM < cu * Rp ? (t + 1) * kTileM : cu * Rp;
                    sfx += (r1 - 1) / Rp - t * kTileM / Rp + 1;
                }
                sfx *= 2 * pl.nh - 1;  // pass 0: every piece; each later pass: one
            }
            const long long units = (long long)((Kq + cu - 1) / cu) * n_instr * dm.Hkv;
            const double boxes = tiles > 1 && cu > 1 ? 0.03 * kTileM / seg : 0.03;
            const double cost = (double)((units + sms - 1) / sms) * (tiles * (pl.nblk + 1 + boxes) + sfx * 1.3);
            if (best < 0.0 || cost < best * 0.97) {
                best = cost;
                pl.Rp = Rp;
                pl.cu = cu;
                pl.cpp = cpp;
                pl.seg = tiles == 1 ? Rp : cu == 1 ? kTileM : seg;
                pl.cbox = tiles == 1 && n_instr == 1 ? cu : 1;  // (a box must not reach into the next instruction)
            }
        }
    }
    {
        // Split: the busiest SM's share is its units times the dearer kind.  Taken where that is well below what whole
        // candidates give, which is when they leave SMs idle: one candidate of 113 tokens, 4 heads per KV head and
        // 78 prefix tokens is 8 units of 20 items on 148 SMs, or 48 units of at most 4 items.
        const int tiles = (round_up(Rg, 8) + kTileM - 1) / kTileM;
        const long long units = (long long)Kq * n_instr * dm.Hkv * (tiles + pl.nh);
        const double dq = pl.nblk + 1 + pl.nh, piece = tiles * 2.3;
        const double cost = (double)((units + sms - 1) / sms) * (dq > piece ? dq : piece);
        pl.n_sub = 1;
        if (tiles <= 1024 && cost < 0.85 * best) {
            pl.n_tiles = tiles;
            pl.n_sub = tiles + pl.nh;
            pl.Rp = round_up(Rg, 8);
            pl.cu = pl.cpp = pl.cbox = 1;
            pl.seg = tiles == 1 ? pl.Rp : kTileM;
        }
    }
    // (a box of one candidate reaches past its last key, where it is filled with zeros)
    pl.sfx_box = pl.nh > 1 ? kPieceN : pl.cpp == 1 ? round_up(pl.Sp, 16) : pl.Sp;
    pl.upi = (Kq + pl.cu - 1) / pl.cu;
    const int slabs = dm.d / 64;
    const int tile_bytes = slabs * kTileM * 128, piece_bytes = slabs * kPieceN * 128;
    pl.terms = dm.S % 8 != 0 || dm.S > kPieceN ? 2 : 1;  // (see the head of this file)
    const int fixed = 2 * tile_bytes + 3 * pl.terms * kDsBytes + kRowsBytes + kBarBytes + 64;
    int n = (kMaxSmem - fixed) / piece_bytes;
    if (n > 2 * kMaxRing) n = 2 * kMaxRing;
    if (n < 2) return pl;
    // a K piece is needed until its dQ product, a V piece only for dP (three and one rather than two and two: see above)
    pl.stages_v = n > 4 ? n / 2 : 1;
    pl.stages_k = n - pl.stages_v;
    pl.off_do = 0;
    pl.off_q = tile_bytes;
    pl.off_k = 2 * tile_bytes;
    pl.off_v = pl.off_k + pl.stages_k * piece_bytes;
    pl.off_p = pl.off_v + pl.stages_v * piece_bytes;
    pl.off_ds = pl.off_p + pl.terms * kDsBytes;
    pl.off_rows = pl.off_ds + 2 * pl.terms * kDsBytes;
    pl.off_bar = pl.off_rows + kRowsBytes;
    pl.off_misc = pl.off_bar + kBarBytes;
    pl.smem_bytes = pl.off_misc + 64;
    pl.ok = pl.smem_bytes <= kMaxSmem && (long long)pl.upi * n_instr * dm.Hkv * pl.n_sub < 2000000000ll;
    return pl;
}

const BwdPlan &plan_bwd(const Dims &dm, int n_instr)
{
    static thread_local PlanTable<BwdPlan> table;
    return table.get(dm, n_instr, [&] { return make_plan(dm, n_instr); });
}

// Where D is formed.
// By the element-wise warps on the smallest launches, whose CTAs have one tile each.  Its loads then run under those of the tile's
// operands, and a launch in the chain of three goes away.  Whole steps, gradients in one term, with the pre-pass and with D in here: 8 candidates, 4/4
// heads, d = 64, P = 32, S = 8 14.1 and 12.0 us; 9, 32/8 heads, P = 256, S = 30 21.8 and 18.2; 2, 32/32 heads, P = 200, S =
// 128 24.3 and 21.6, P = 300, S = 50 21.7 and 21.2.  With several tiles per CTA every tile waits for its own D: 1
// candidate, 32/8 heads, P = 78, S = 113 (four tiles in a unit) 25.3 and 28.8, 12 candidates, 32/32 heads, P = 90, S = 77
// (three units per CTA) 38.7 and 43.9.
// As an item of its own on larger ones: 512 MMA cycles and one hand-off per tile instead of a pass over dout and out at the rate
// of HBM and its launch.  Whole steps, pre-pass and item: 512 candidates, 32/8 heads, P = 256, S = 48 528 and 510 us, 8 x 64 in instructions 525 and
// 508; 49, 32/8, P = 108, S = 47 57 and 53; with one tile to a unit on launches of few units 46, 32/32, P = 77, S = 20 45.6 and 43.8; 16,
// P = 100, S = 55 40.6 and 37.6.
// What it needs: head dim 128, no gradient on lse, units that are no parts of a candidate, and suffix boxes of whole steps of 16 keys (the
// MMAs read K and V stages in such steps, and `out` passes through the same stages: nothing of it must be left to be read).
// Where it is not taken, and what is known of both there:
//  - `out` in boxes below 24 rows: 500, 32/32, P = 211, S = 10 (16 rows) 209 and 219.
//  - one tile to a unit from four units per SM on: 60, 32/32, P = 256, S = 47 (960 units) 115 and 121; 400, 32/16, P = 100, S = 51 453 and
//    459; 250, 32/8, P = 100, S = 21 115 and 121; 314, 32/32, P = 635, S = 19 368 and 374; no difference for 128, P = 160 to 2048, S = 40.  Only full
//    tiles of one term gain: 256, 32/8, S = 32, P = 128 to 2048 134, 255, 412, 724 and 127, 246, 405, 722.
//  - two terms, one candidate to a unit whose tiles are at most seven eighths full, two prefix pieces, from four units per SM on: the item
//    works on whole tiles, the pass on rows, and three items of two terms and one V stage do not cover the hand-off.  250, 32/8, P = 100, S = 49,
//    51, 55, 57, 61 255, 263, 278, 292, 300 and 261, 268, 281, 289, 294; 300, P = 65, S = 50 303 and 314; 70, P = 100, S = 51 80.0 and 79.1; with one prefix
//    piece (333, P = 32, S = 53) 305 and 299, with three (250, P = 129, S = 51) 307 and 301.
//  - suffixes of several pieces.  Tiles of a unit of several are walked over once per piece, and each time D is formed again: 44, 32/8, P = 51, S =
//    87 113 and 120.  Units of one tile are walked over once; from four units per SM on they lose (40, 32/32, P = 500, S = 72 167 and 172; 34, P = 136,
//    S = 96 107 and 111; 28, P = 75, S = 69 76.8 and 79.5; 304 in 8 instructions, P = 512, S = 80 1271 and 1334), below that they would gain
//    (8, P = 78, S = 113 40 and 36; 18, P = 300, S = 100 81 and 79; 6, P = 50, S = 111 37 and 33).
//  - several instructions below four units per SM.  These calls are known, and tested, as two launches, one for the row statistic and one
//    for the gradients; the item in front of theirs is faster (64 candidates in 2 instructions, 32/8, P = 256, S = 48 75.5 and 72.9; 16 in 4, 32/32,
//    P = 150, S = 55 43.3 and 40.2; 128 in 4, 32/8, P = 128, S = 48 115 and 110).
DSource d_source(const BwdArgs &a, const BwdPlan &plan, int n_instr)
{
    const Dims &dm = a.dims;
    const long long units = (long long)plan.upi * n_instr * dm.Hkv * plan.n_sub;
    const int tiles = (plan.cu * plan.Rp + kTileM - 1) / kTileM;
    if (n_instr == 1 && tiles == 1 && units <= sm_count()) return kDWarps;
    const bool can = dm.d == 128 && !a.dlse && plan.n_sub == 1 && plan.sfx_box * plan.cpp % 16 == 0;
    if (!can || plan.nh > 1 || plan.seg * plan.cbox < 24) return kDTable;
    if (units < 4ll * sm_count()) return n_instr == 1 ? kDItem : kDTable;
    const bool part_full = plan.terms == 2 && plan.cu == 1 && plan.nblk == 2 && 8 * plan.Rp <= 7 * kTileM * tiles;
    return tiles == 1 || part_full ? kDTable : kDItem;
}

template <int D, bool TWO>
cudaError_t launch(const BwdArgs &a, const BwdPlan &plan, unsigned int *status_word, cudaStream_t stream, int n_instr,
                   const int *prefix_len, DSource dsrc)
{
    const Dims &dm = a.dims;
    const int Rg = dm.n_rep * dm.S;
    CUtensorMap tm_q, tm_do, tm_pk, tm_pv, tm_sk, tm_sv, tm_out;
    memset(&tm_out, 0, sizeof(tm_out));
    memset(&tm_pk, 0, sizeof(tm_pk));
    memset(&tm_pv, 0, sizeof(tm_pv));
    {
        // q / dout viewed as [B][Hkv][Rg][D]: the n_rep heads of a KV head are contiguous rows.  A box that
        // reaches past a candidate's last row reads zeros there.
        cuuint64_t dims[4] = {(cuuint64_t)D, (cuuint64_t)Rg, (cuuint64_t)dm.Hkv, (cuuint64_t)dm.B};
        cuuint64_t str[3] = {(cuuint64_t)D * 2, (cuuint64_t)Rg * D * 2, (cuuint64_t)dm.Hkv * Rg * D * 2};
        cuuint32_t box[4] = {64, (cuuint32_t)plan.seg, 1, (cuuint32_t)plan.cbox};
        if (!encode_map(&tm_q, a.q, 4, dims, str, box)) return cudaErrorInvalidValue;
        if (!encode_map(&tm_do, a.dout, 4, dims, str, box)) return cudaErrorInvalidValue;
        if (dsrc == kDItem && !encode_map(&tm_out, a.out, 4, dims, str, box)) return cudaErrorInvalidValue;
    }
    {
        cuuint64_t dims[4] = {(cuuint64_t)D, (cuuint64_t)dm.S, (cuuint64_t)dm.Hkv, (cuuint64_t)dm.B};
        cuuint64_t str[3] = {(cuuint64_t)D * 2, (cuuint64_t)dm.S * D * 2, (cuuint64_t)dm.Hkv * dm.S * D * 2};
        cuuint32_t box[4] = {64, (cuuint32_t)plan.sfx_box, 1, (cuuint32_t)plan.cpp};
        if (!encode_map(&tm_sk, a.suffix_k, 4, dims, str, box)) return cudaErrorInvalidValue;
        if (!encode_map(&tm_sv, a.suffix_v, 4, dims, str, box)) return cudaErrorInvalidValue;
    }
    if (dm.P > 0) {
        cuuint64_t dims[3] = {(cuuint64_t)D, (cuuint64_t)dm.P, (cuuint64_t)dm.Hkv * (cuuint64_t)n_instr};
        cuuint64_t str[2] = {(cuuint64_t)D * 2, (cuuint64_t)dm.Pstride * D * 2};
        cuuint32_t box[3] = {64, (cuuint32_t)kPieceN, 1};
        if (!encode_map(&tm_pk, a.prefix_k, 3, dims, str, box)) return cudaErrorInvalidValue;
        if (!encode_map(&tm_pv, a.prefix_v, 3, dims, str, box)) return cudaErrorInvalidValue;
    }
    TcBwdParams p;
    memset(&p, 0, sizeof(p));
    p.lse = a.lse;
    p.row_dot = a.row_dot;
    p.out = a.out;
    p.dout = a.dout;
    p.dlse = a.dlse;
    p.dq = a.dq;
    p.dq_two = dm.S % 8 != 0 || dm.S > kTileM;
    p.dq_sectors = (reinterpret_cast<uintptr_t>(a.dq) & 31u) == 0;
    p.dk = a.dk_suffix;
    p.dv = a.dv_suffix;
    p.status = status_word;
    p.sl2 = a.scale * kLog2e;
    p.scale = a.scale;
    p.Hq = dm.Hq; p.Hkv = dm.Hkv; p.S = dm.S; p.P = dm.P; p.n_rep = dm.n_rep;
    p.Rg = Rg; p.Rp = plan.Rp; p.Sp = plan.Sp;
    p.cu = plan.cu; p.cpp = plan.cpp; p.nh = plan.nh; p.seg = plan.seg; p.cbox = plan.cbox; p.sfx_box = plan.sfx_box;
    p.nblk = plan.nblk;
    p.Kq = dm.B / n_instr;
    p.upi = plan.upi;
    p.upg = plan.upi * n_instr;
    p.fd_upg.init(p.upg);
    p.fd_upi.init(p.upi);
    p.n_tiles = plan.n_tiles;
    p.n_sub = plan.n_sub;
    p.fd_sub.init(p.n_sub);
    p.fd_Rp.init(p.Rp);
    p.fd_S.init(dm.S);
    p.fd_cpp.init(p.cpp);
    p.stages_k = plan.stages_k; p.stages_v = plan.stages_v;
    p.off_do = plan.off_do; p.off_q = plan.off_q; p.off_k = plan.off_k; p.off_v = plan.off_v; p.off_p = plan.off_p;
    // The MMAs contract over rows and keys in steps of 16: boxes of a multiple of 16 rows (keys) leave none unwritten.
    p.zero_lo = plan.seg * plan.cbox % 16 != 0 ? plan.off_do : plan.off_k;
    p.zero_hi = plan.sfx_box * plan.cpp % 16 != 0 ? plan.off_p : plan.off_k;
    p.off_ds = plan.off_ds; p.off_rows = plan.off_rows; p.off_bar = plan.off_bar; p.off_misc = plan.off_misc;
    for (int i = 0; i < n_instr && n_instr > 1; ++i) p.pad[i] = dm.P - prefix_len[i];

    const bool sp = plan.n_sub > 1;
    auto kernel = sp ? tc_bwd_kernel<D, true, kDTable, TWO> : tc_bwd_kernel<D, false, kDTable, TWO>;
    if (dsrc == kDWarps) kernel = sp ? tc_bwd_kernel<D, true, kDWarps, TWO> : tc_bwd_kernel<D, false, kDWarps, TWO>;
    if constexpr (D == 128)
        if (dsrc == kDItem) kernel = tc_bwd_kernel<D, false, kDItem, TWO>;
    static PerDeviceOnce attr_set[6];
    if (cudaError_t e = ensure_max_smem(kernel, attr_set[2 * dsrc + sp]); e != cudaSuccess) return e;
    p.n_units = p.upg * dm.Hkv * p.n_sub;
    cudaError_t e;
    {
        KernelTiming timing(kKernelBwdTc, stream);
        e = launch_dependent(kernel, even_grid(p.n_units, sm_count()), kThreads, plan.smem_bytes, stream, tm_q, tm_do, tm_pk, tm_pv,
                             tm_sk, tm_sv, tm_out, p);
    }
    count_launches(1);
    return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace

#ifdef PSKV_TRACE
// Debug builds only: copies this kernel's event trace of one CTA to the host.
extern "C" int pskv_debug_read_trace_bwd(long long *host, int max_events)
{
    static long long buf[kTraceWarps * kTraceCap * 2];
    unsigned int cnt[kTraceWarps];
    cudaDeviceSynchronize();
    cudaMemcpyFromSymbol(cnt, g_trace_n, sizeof(cnt));
    cudaMemcpyFromSymbol(buf, g_trace, sizeof(buf));
    int n = 0;
    for (int w = 0; w < kTraceWarps; ++w)
        for (unsigned int i = 0; i < cnt[w] && i < (unsigned int)kTraceCap && n < max_events; ++i, ++n) {
            host[2 * n] = buf[((size_t)w * kTraceCap + i) * 2];
            host[2 * n + 1] = buf[((size_t)w * kTraceCap + i) * 2 + 1] | ((long long)w << 24);
        }
    return n;
}
#endif

bool tc_bwd_supported(const Dims &dm)
{
    if (dm.Skv != dm.S || dm.ragged) return false;  // full-suffix operator only
    if (dm.d != 64 && dm.d != 128) return false;
    if ((long long)dm.B * dm.n_rep * dm.S > 2000000000ll || dm.n_rep * (long long)dm.S > 1000000ll) return false;
    return plan_bwd(dm, 1).ok && get_encode_fn() != nullptr;
}

size_t tc_bwd_workspace_bytes(const Dims &dm) { return (size_t)dm.B * dm.Hq * dm.S * sizeof(float); }

bool tc_bwd_fused_supported(const Dims &dm, int n_instr)
{
    return n_instr >= 2 && n_instr <= kMaxFusedInstructions && dm.B % n_instr == 0 && dm.P >= 1 && dm.Pstride == dm.P &&
           tc_bwd_supported(dm) && plan_bwd(dm, n_instr).ok;
}

cudaError_t launch_tc_bwd(const BwdArgs &a, unsigned int *status_word, cudaStream_t stream, int parts, int n_instr,
                          const int *prefix_len)
{
    if (n_instr < 1) n_instr = 1;
    if (n_instr > 1 && (!prefix_len || !tc_bwd_fused_supported(a.dims, n_instr))) return cudaErrorInvalidValue;
    const BwdPlan &plan = plan_bwd(a.dims, n_instr);
    if (!plan.ok) return cudaErrorInvalidValue;
    const DSource dsrc = parts == kBwdPartAll ? d_source(a, plan, n_instr) : kDTable;
    if ((parts & kBwdPartRowDot) && dsrc == kDTable) {
        const cudaError_t e = launch_simt_row_dot(a, stream);
        if (e != cudaSuccess) return e;
    }
    if (!(parts & kBwdPartGrad)) return cudaSuccess;
    auto run = plan.terms == 2 ? (a.dims.d == 128 ? launch<128, true> : launch<64, true>)
                               : (a.dims.d == 128 ? launch<128, false> : launch<64, false>);
    return run(a, plan, status_word, stream, n_instr, prefix_len, dsrc);
}

}  // namespace pskv
