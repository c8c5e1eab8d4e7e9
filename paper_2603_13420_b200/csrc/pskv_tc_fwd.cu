// Fused shared-prefix attention forward for sm_100a (tcgen05 / TMEM / TMA).
//
// All B*(Hq/Hkv)*S query rows of one KV head form one long row list that is cut into tiles of
// up to 128 rows; each tile is one dense contraction against the single shared prefix K/V of
// that KV head (kept in shared memory across tiles when it fits, never copied per candidate,
// Sec. 4.2), followed by one block holding the suffix keys of the few candidates the tile
// touches (block-diagonal causal mask).  Scores go to tensor memory, one continued online
// softmax runs over prefix blocks and the suffix block (Eq. 2; equivalent to merging the two
// partial results by their log-sum-exp), probabilities go back to tensor memory as bf16 and are
// the A operand of the P*V contraction; `out` and `lse` are written once.
//
// Persistent CTA, one per SM, 24 warps:
//   warp 0      TMA producer, score side (Q tile, prefix K blocks, suffix K of the tile)
//   warp 1      tcgen05.mma issuer for the score blocks  S = Q K^T
//   warp 2      tcgen05.mma issuer for the value blocks  O += P V   (owns the TMEM allocation)
//   warp 3      TMA producer, value side (prefix V blocks, suffix V of the tile); TMA stores of `out`
//   warps 4-19  softmax, four warpgroups sharing each item by 32-column pieces (thread <-> query
//               row = TMEM lane)
//   warps 20-23 epilogue: O / row sum -> bf16 -> staging buffer, lse
// An "item" is one (tile, key block) pair; tensor memory holds three 128-column score slots (the
// bf16 probabilities of an item overwrite parts of its own slot) and the 128 columns of O.  Every
// wait is on an event produced by an earlier item of a role that never waits on the waiter, so
// no wait cycle can form; every wait is bounded.
//
// Three instantiations share this code (see the comment at the kernel): prefix streamed through
// rings, prefix resident in shared memory, and the suffix-ring mode, in which a tile is a run of
// whole candidates (or of rows inside one candidate) and the suffix keys follow the prefix through
// the same rings in as many blocks as it takes -- the mode of the decode-shaped operator, of
// suffixes beyond one key block and of the causal self-attention of a single sequence.
#include <string.h>

#include "pskv_common.cuh"
#include "pskv_rows.cuh"
#include "pskv_sm100.cuh"
#include "pskv_tc_common.cuh"

namespace pskv {
namespace {

using namespace sm100;

constexpr int kSlots = 3;      // score slots of 128 columns; an item's probabilities overwrite its own scores
constexpr int kGroups = 4;     // softmax warpgroups: one 32-column piece of every score block each
constexpr int kThreads = 32 * (4 + 4 * kGroups + 4);
constexpr int kOCol = kSlots * kBlockN;  // first tensor-memory column of O
// Probabilities are 2^(s * sl2) with no max subtracted; rows whose sum leaves
// [kMinRowSum, kMaxRowSum] are redone with max subtraction at the end of the kernel.
constexpr float kMaxRowSum = 1.2676506002282294e30f;   // 2^100
constexpr float kMinRowSum = 7.8886090522101181e-31f;  // 2^-100
constexpr int kMaxStages = 4;
constexpr int kMaxInstr = kMaxFusedInstructions;  // prefixes one launch can serve

enum : unsigned int {
    kErrProducerK = 0x101, kErrProducerV = 0x102, kErrMmaQk = 0x103, kErrMmaPv = 0x104,
    kErrSoftmax = 0x105, kErrEpilogue = 0x106, kErrAlign = 0x107
};

// MODE 3.  The compiler reads runs of the kernel's parameters in one instruction where they are aligned, and what that makes of the
// walk over tiles differs.  The fields behind these moved by 12 bytes and by 16: several instructions of whole tiles, prefix resident, 8 x 64
// candidates, 32/8 heads, P = 256, S = 48 178 and 160 us, 4 x 32, P = 128 38.5 and 35.3; streamed, 6 x 60, P = 300, S = 40 130 and 136; short last
// tiles, 6 x 90, P = 300, S = 37 196 and 198; one prefix, 333, P = 217, S = 53 119 and 116, 149, 4/4, P = 315, S = 8 10.4 both.
template <bool ALIGNED>
struct BoxFields {
    int Sh;               // rows a query head takes in the row list: S, or S padded to whole tiles (head_box)
    int one_box;          // 1: a tile's Q is one box per slab (whole candidates, or rows of one head), else runs of seg_rows
    int head_box;         // 1: Q / out maps are [B][Hq][S][D] and a tile lies inside one head
};
template <>
struct BoxFields<true> {
    int Sh, one_box, head_box, unused;
};

template <int MI>
struct TcFwdParams {
    float *lse;
    unsigned int *status;
    FwdArgs args;         // the call's raw arguments, for the rows that are redone row by row
    float sl2;            // scale * log2(e)
    int B, Hq, Hkv, S, P, n_rep;
    int Rg;               // rows a candidate takes in the row list of a KV-head group (its n_rep * S real rows, padded)
    int Rr;               // its real rows: n_rep * S
    int Sp;               // key columns a candidate takes in a tile's suffix block: S rounded up to 8
    BoxFields<MI == 1> box;
    int tile_rows;        // rows of the flat row list per tile (<= 128, multiple of seg_rows)
    int seg_rows;         // rows per Q / out TMA box: gcd(Rg, tile_rows) (rows past Rr are zero-filled, never stored)
    int tiles_per_group;
    FastDiv fd_tpg, fd_Rg, fd_S, fd_seg;  // divisions by tiles_per_group, Rg, Sh, seg_rows
    int total_tiles;
    int nblk_p;           // prefix key blocks: ceil(P / 128)
    int tail_rows;        // rows held by the last prefix block (multiple of 16, <= 128)
    int resident;         // 1 when all prefix blocks of a KV head stay in shared memory
    int stages;           // streaming mode: stages of the prefix K and V rings
    int sfx_rows;         // rows of the suffix K / V buffers (multiple of 16, <= 128)
    int alias_stage;      // 1 when the output staging buffer shares its memory with the suffix V buffer
    int slab_stage;       // 1 when the staging buffer holds one 64-column slab: staged and stored a slab at a time
    int ml_mask;          // partial row sums are kept for ml_mask + 1 tiles (3, or 0 behind kBarMlFree)
    // suffix-ring mode (tiles of whole candidates, suffix keys in blocks through the K/V rings)
    const int *suffix_len;  // cached suffix tokens per candidate, or nullptr (= Skv)
    int Skv;              // rows of a candidate's suffix K/V buffer (S counts its query rows)
    int Spad;             // Skv rounded up to 8: rows a candidate takes inside a suffix block
    int cpb;              // candidates per suffix block: 128 / Spad
    FastDiv fd_cpb;
    int deal_by_cost;     // long suffixes: hand tiles to CTAs by cost rank instead of in contiguous ranges
    int long_sfx;         // 1: a tile lies inside ONE candidate and that candidate's suffix keys come in
                          //    128-key blocks (suffix caches or row groups beyond 128); 0: whole-candidate tiles
    // several instructions in one launch (Sec. 4.3): the candidates of instruction i are contiguous and use
    // prefix cache i of [n_instr][Hkv][P][d], whose first pad[i] rows are left padding
    int n_instr;          // 1: one shared prefix
    int rpi;              // rows of one instruction inside a KV head's row list
    FastDiv fd_rpi, fd_tpi;
    int tpi;              // tiles of an instruction, where each starts a tile of its own and its last tile is short
    int pad[kMaxInstr];
    // shared-memory carve-up (byte offsets from the 1024-byte aligned base)
    int off_pk, off_pv, off_q, off_sk, off_sv, off_stage, off_bar, off_misc, off_ml;
    int zero_lo, zero_hi;  // V buffers whose rows no copy may reach before the value MMAs read them
};

template <int D>
struct Cfg {
    static constexpr int kSlabs = D / 64;              // 64-column (128-byte) swizzle slabs per row
    static constexpr int kSlabBytes = kTileM * 128;    // a full slab: 128 rows x 128 bytes
    static constexpr int kTileBytes = kSlabs * kSlabBytes;
};

// barrier indices
enum {
    kBarQFull = 0,   // Q tile landed
    kBarQkFree,      // all score MMAs of a tile completed: Q and suffix-K buffers are free
    kBarSKFull,
    kBarSVFull,
    kBarSVFree,      // all value MMAs of a tile completed: suffix-V buffer is free
    kBarOFull,       // O of a tile is complete in tensor memory
    kBarOFree,       // epilogue has read O out (one arrival per softmax warp)
    kBarStageFull,   // the output tile is staged (one arrival per softmax warp)
    kBarStageFree,   // the TMA stores of that slab have read it
    kBarMlFree,      // the epilogue has read a tile's partial row sums (one arrival per epilogue warp)
    kBarSFull,                        // [kSlots] scores of an item are in tensor memory
    kBarPReady = kBarSFull + kSlots,  // [kSlots] probabilities written (one arrival per softmax warp)
    kBarPvDone = kBarPReady + kSlots, // [kSlots] value MMAs of an item completed
    kBarKFull = kBarPvDone + kSlots,  // [stages]
    kBarVFull = kBarKFull + kMaxStages,
    kBarKFree = kBarVFull + kMaxStages,
    kBarVFree = kBarKFree + kMaxStages,
    kNumBars = kBarVFree + kMaxStages
};
constexpr int kBarBytes = 512;
static_assert(kNumBars * 8 <= kBarBytes, "barrier area");

// Q / out box coordinates of row r of a group: (row, head) -- the group's row list seen as one head, or the head itself
template <bool ANY, class Params>
__device__ __forceinline__ void q_coords(const Params &p, int r, int g, int &c1, int &c2)
{
    c1 = r;
    c2 = g;
    if (ANY && p.box.head_box) {
        const int h = p.fd_S.div(r);
        c1 = r - h * p.box.Sh;
        c2 = g * p.n_rep + h;
    }
}

// rows held (and MMA N used) by prefix block k
template <class Params>
__device__ __forceinline__ int prefix_block_rows(const Params &p, int k)
{
    return k == p.nblk_p - 1 ? p.tail_rows : kBlockN;
}

constexpr int kPiece = 32;  // score columns a softmax thread handles per tensor-memory load
static_assert(kBlockN == 4 * kPiece, "two softmax groups x two pieces cover a score block");

// Suffix-ring mode: candidates [first, first + count) of a tile that suffix block j holds, and the
// MMA N (rows rounded up to 16) of that block.
template <class Params>
__device__ __forceinline__ int sfx_block_cands(const Params &p, int nc, int j)
{
    return min(p.cpb, nc - j * p.cpb);
}
template <class Params>
__device__ __forceinline__ int sfx_block_rows(const Params &p, int nc, int j)
{
    return (sfx_block_cands(p, nc, j) * p.Spad + 15) & ~15;
}

// Suffix-ring mode with long suffixes: the tile's rows belong to one candidate; it needs that
// candidate's suffix keys up to the last one any of its rows may see, in blocks of 128.
template <bool ANY, class Params>
__device__ __forceinline__ int sfx_blocks_long(const Params &p, const TileInfo &t)
{
    const int r0 = t.R0 - t.b_first * p.Rg;
    const int s0 = r0 - p.fd_S.div(r0) * (ANY ? p.box.Sh : p.S);  // query index of the tile's first row
    const int s_max = (s0 + t.rows > p.S) ? p.S - 1 : s0 + t.rows - 1;  // rows wrap into the next head
    const int pos = suffix_tokens(p.suffix_len, t.b_first, p.S, p.Skv) - p.S + s_max;
    return (pos >> 7) + 1;
}
// MMA N of long-suffix block j (its 128-row box is zero-filled past the end of the cache)
template <class Params>
__device__ __forceinline__ int sfx_long_rows(const Params &p, int j)
{
    return min(kBlockN, (p.Skv - j * kBlockN + 15) & ~15);
}

// MODE 1: all prefix blocks of a KV head stay in shared memory; MODE 0: they stream through rings,
// and the suffix keys of a tile sit in one block with buffers of its own; MODE 2 and 3 (suffix-ring): the suffix
// keys follow the prefix through the same rings in as many blocks as it takes.  MODE 2: a tile lies inside one
// candidate, whose rows the tiles divide (suffix caches beyond a block, prompts); MODE 3: any row list -- whole candidates
// (the decode-shaped operator, where a 128-row tile spans many), tiles that straddle candidates, tiles inside a head
// whose rows are padded to whole tiles.  A compile-time
// switch so that each launch carries only the code of its own mode.  The last two are apart for what the compiler makes of
// them: 729 beams, 32/32 heads, 4 tokens over 147 cached ones take 572 us in MODE 2 and 644 with MODE 3's decisions at run time,
// 512 beams, 32/8 heads, one token over 48 23.8 us in MODE 3 and 25.6 with MODE 2's code.
// MI 1: several instructions, each a whole number of tiles; 2: the last tile of each is short.  Apart because a tile's
// place is worked out by every role (8 x 64 candidates, 32/8 heads, P = 256, S = 48: 139 us with the second's division, 132).
//
// TWO (MODE 3): probabilities as the sum of two bf16 values, the second in the half of a piece that the first leaves free, and
// a value contraction over each.  For the lengths that came from the CUDA-core kernel (two_terms in plan_suffix_ring), whose
// probabilities are fp32.  Distance (2-norm) of `out` from 64 bits, a prompt of 1039 tokens, 32/8 heads: CUDA cores 1.625e-3,
// one term 2.310e-3, two terms 1.625e-3 (the rounding of the result); of lse 4.9e-8, 7.6e-8 and, with the logarithm in 64
// bits, 4.1e-8 (131 tokens: 4.8e-8, 8.0e-8 and 5.4e-8: what is left is the tensor cores' fp32 sum of a score; one rounding of
// the result is 2.7e-8).  Price: 131 tokens 8.7 -> 9.0 us, 1039 21.0 -> 24.0, 4093 131 -> 170 (CUDA cores 52 us, 1.58 and
// 22.2 ms).
template <int D, int MODE, int MI, bool TWO = false>
__global__ void __launch_bounds__(kThreads, 1)
tc_fwd_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_out,
              const __grid_constant__ CUtensorMap tm_pk, const __grid_constant__ CUtensorMap tm_pv,
              const __grid_constant__ CUtensorMap tm_pk_tail, const __grid_constant__ CUtensorMap tm_pv_tail,
              const __grid_constant__ CUtensorMap tm_sk, const __grid_constant__ CUtensorMap tm_sv,
              const TcFwdParams<MI> p)
{
    using C = Cfg<D>;
    constexpr bool RES = MODE == 1;
    constexpr bool SR = MODE >= 2, ANY = MODE == 3;
    constexpr bool PAD = MODE != 2;  // a candidate's rows may be followed by rows that do not exist
    extern __shared__ __align__(1024) uint8_t smem[];
    const int tid = threadIdx.x, lane = tid & 31;
    const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);  // warp-uniform by construction
    PSKV_TRACE_DECL;
    grid_dep_launch();  // the next kernel of the stream may take over SMs as this one's CTAs exit
    const uint32_t sbase = smem_u32(smem);
    const uint32_t bar0 = sbase + p.off_bar;
    auto bar = [&](int i) { return bar0 + 8u * (uint32_t)i; };
    volatile int *abort_flag = reinterpret_cast<volatile int *>(smem + p.off_misc + 4);
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(smem + p.off_misc);
    int *cta_redo = reinterpret_cast<int *>(smem + p.off_misc + 8);  // rows of this CTA's tiles to redo
    float *ml = reinterpret_cast<float *>(smem + p.off_ml);  // partial row sums [tile % 4][softmax group][128]

    if ((sbase & 1023u) != 0u) {  // the swizzled layouts need a 1024-byte aligned base
        if (tid == 0) atomicCAS(p.status, 0u, (unsigned int)kErrAlign);
        return;
    }

    // Value rows that no TMA box ever writes must hold finite values, because a zero probability times a NaN would
    // still poison the accumulator.  Q and K rows need nothing: what they lead to is masked or never stored.
    // (With all 220 KB zeroed by every launch, and the barriers set up by one thread in front of a second block
    // barrier, launches behind a kernel that gives their prologue no cover took 53.4 us instead of 51.8 for a
    // causal pass over 2048 tokens, 43.2 instead of 41.5 for 40 candidates, 32/32 heads, P = 700, S = 37.)
    for (int i = p.zero_lo / 16 + tid; i < p.zero_hi / 16; i += kThreads)
        reinterpret_cast<uint4 *>(smem)[i] = make_uint4(0, 0, 0, 0);
    if (warp == 3) {
        for (int i = lane; i < kNumBars; i += 32) {
            const bool all_sm = i >= kBarPReady && i < kBarPReady + kSlots;
            const bool epi = i == kBarOFree || i == kBarStageFull || i == kBarMlFree;
            mbar_init(bar(i), all_sm ? (uint32_t)(4 * kGroups) : epi ? 4u : 1u);
        }
        if (lane == 0) {
            *abort_flag = 0;
            *cta_redo = 0;
        }
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

    // Tiles of this CTA.  Normally a contiguous range (tiles are ordered KV head major, so the
    // resident prefix of a head serves a whole run).  With long suffixes a tile's cost grows with the
    // position of its rows inside the suffix (causal block skipping), so there -- when tiles do not
    // straddle heads and the suffix K/V of all candidates stays in L2 anyway -- the tiles are dealt out by cost: ranked from the last (longest) suffix
    // position down, round r hands ranks r*G .. r*G+G-1 to the CTAs in alternating direction (the
    // longest-first rule in closed form).
    const int t_begin = (int)((long long)blockIdx.x * p.total_tiles / gridDim.x);
    const int t_end = (int)((long long)(blockIdx.x + 1) * p.total_tiles / gridDim.x);
    const int G = (int)gridDim.x;
    const int Sh = ANY ? p.box.Sh : p.S;
    // What MODE 2 knows of its plan: with these decided at run time it spilled 12 registers (396 bytes of loads; 20 candidates, 32/8
    // heads, P = 64, S = 300 58 us, now 53).
    const bool long_sfx = MODE == 2 || p.long_sfx;
    const bool slab_stage = MODE != 2 && p.slab_stage, alias_stage = MODE != 2 && p.alias_stage;
    const int n_sp = (SR && p.deal_by_cost) ? Sh / p.tile_rows : 1;  // tiles per head
    const bool dealt = n_sp > 1;
    auto rank_at = [&](int tl) { return tl * G + ((tl & 1) ? G - 1 - (int)blockIdx.x : (int)blockIdx.x); };
    auto tile_at = [&](int tl) {
        if (!dealt) return t_begin + tl;
        // rank -> (suffix position from the end, candidate, KV head, head inside the group)
        const int rank = rank_at(tl), M = p.B * p.Hkv * p.n_rep;
        const int spr = rank / M, m = rank - spr * M;
        const int b = m / (p.Hkv * p.n_rep), gh = m - b * (p.Hkv * p.n_rep);
        const int g = gh / p.n_rep, hr = gh - g * p.n_rep;
        return g * p.tiles_per_group + (b * p.n_rep + hr) * n_sp + (n_sp - 1 - spr);
    };
    const int n_rounds = (p.total_tiles + G - 1) / G;
    const int n_tiles = !dealt ? t_end - t_begin : (n_rounds - 1) + (rank_at(n_rounds - 1) < p.total_tiles ? 1 : 0);
    // items of a tile: prefix blocks + the suffix block(s)
    auto items_of = [&](const TileInfo &t) {
        return p.nblk_p + (!SR ? 1 : long_sfx ? sfx_blocks_long<ANY>(p, t) : p.fd_cpb.div(t.nc + p.cpb - 1));
    };
    // A run of tiles that shares one prefix: a KV head, or (several instructions) one instruction's
    // candidates inside a KV head.  Runs are numbered in tile order; the resident prefix is reloaded at the
    // start of each run and the barrier parity of those loads follows the run number.
    auto inst_of = [&](const TileInfo &t) { return MI ? p.fd_rpi.div(t.R0) : 0; };
    auto run_of = [&](const TileInfo &t, int inst) { return MI ? t.g * p.n_instr + inst : t.g; };
    auto first_of_run = [&](const TileInfo &t, int inst) {
        return t.first_of_g || (MI && t.R0 == inst * p.rpi);
    };
    // First prefix block a tile works on: the blocks that hold nothing but left padding are skipped by
    // every role (the resident copy still holds them, so the block index stays absolute).
    auto first_block = [&](int inst) { return MI ? p.pad[inst] / kBlockN : 0; };
    int run_first;
    {
        const TileInfo t0 = tile_info<MI == 2>(p, t_begin < p.total_tiles ? t_begin : 0, t_begin);
        run_first = run_of(t0, inst_of(t0));
    }
    const int sfx_slab = p.sfx_rows * 128;
    const int tail_slab = p.tail_rows * 128;

    // The producer and MMA warps run their loops with all 32 lanes (warp-uniform control flow and
    // addresses, so descriptors can live in uniform registers); one elected lane issues the
    // asynchronous instructions.
    const int role = warp;
    if (role == 0) {
        // ------------------------------------------------------------------ producer, score side
        if (lane == 0) {
            prefetch_tensormap(&tm_q);
            prefetch_tensormap(&tm_sk);
            if (p.P > 0) { prefetch_tensormap(&tm_pk); prefetch_tensormap(&tm_pk_tail); }
        }
        uint32_t ks = 0, kph = 1;  // ring of K blocks: stage, parity of its release
        bool ok = true;
#pragma unroll 1
        for (int tl = 0; tl < n_tiles && ok; ++tl) {
            const TileInfo t = tile_info<MI == 2>(p, tile_at(tl), t_begin);
            // Everything the Q loads need is worked out before the wait, so that only the copy
            // instructions themselves follow it: the Q buffer is single, and the time from "last
            // score MMA of the previous tile done" to "Q of this tile requested" is exposed.
            // (Suffix-ring mode: one box per slab holds the tile's whole candidates; a box reaching
            // past the last candidate is filled with zeros and still counts its full size.)
            const int nseg = (SR && (!ANY || p.box.one_box)) ? 1 : p.fd_seg.div(t.rows);  // one box per run of seg_rows rows
            int qb = p.fd_Rg.div(t.R0), qr = t.R0 - qb * p.Rg;
            const uint32_t q_bytes = (uint32_t)(nseg * C::kSlabs * p.seg_rows * 128);
            const uint32_t seg_bytes = (uint32_t)(p.seg_rows * 128);
            uint32_t q_dst = sbase + p.off_q;
            // Q, suffix K and (resident mode) the prefix K blocks are free once every score MMA of
            // the previous tile has completed
            ok = mbar_wait_warp(bar(kBarQkFree), (tl & 1) ^ 1, abort_flag, p.status, kErrProducerK);
            if (!ok) break;
            PSKV_TRACE_EVENT(1, tl);
            if (elect_one_sync()) {
                mbar_arrive_expect_tx(bar(kBarQFull), q_bytes);
#pragma unroll 1
                for (int s = 0; s < nseg; ++s) {
                    int c1, c2;
                    q_coords<ANY>(p, qr, t.g, c1, c2);
#pragma unroll
                    for (int sl = 0; sl < C::kSlabs; ++sl)
                        tma_load_4d(q_dst + sl * C::kSlabBytes, &tm_q, bar(kBarQFull), sl * 64, c1, c2, qb);
                    q_dst += seg_bytes;
                    qr += p.seg_rows;  // boxes never straddle a candidate: seg_rows divides Rg
                    if (qr >= p.Rg) {
                        qr -= p.Rg;
                        ++qb;
                    }
                }
            }
            __syncwarp();
            const int inst = inst_of(t);
            const int ph = inst * p.Hkv + t.g;  // head index inside the prefix caches
            if (RES) {
                if (first_of_run(t, inst) && elect_one_sync()) {
#pragma unroll 1
                    for (int k = 0; k < p.nblk_p; ++k) {
                        const bool tail = k == p.nblk_p - 1;
                        const int slab = tail ? tail_slab : C::kSlabBytes;
                        mbar_arrive_expect_tx(bar(kBarKFull + k), (uint32_t)(C::kSlabs * slab));
#pragma unroll 1
                        for (int sl = 0; sl < C::kSlabs; ++sl)
                            tma_load_3d(sbase + p.off_pk + k * C::kTileBytes + sl * slab, tail ? &tm_pk_tail : &tm_pk,
                                        bar(kBarKFull + k), sl * 64, k * kBlockN, ph);
                    }
                }
                __syncwarp();
            } else {
#pragma unroll 1
                for (int k = first_block(inst); k < p.nblk_p; ++k) {
                    ok = mbar_wait_warp(bar(kBarKFree + ks), kph, abort_flag, p.status, kErrProducerK);
                    if (!ok) break;
                    const bool tail = k == p.nblk_p - 1;
                    const int slab = tail ? tail_slab : C::kSlabBytes;
                    if (elect_one_sync()) {
                        mbar_arrive_expect_tx(bar(kBarKFull + ks), (uint32_t)(C::kSlabs * slab));
#pragma unroll 1
                        for (int sl = 0; sl < C::kSlabs; ++sl)
                            tma_load_3d(sbase + p.off_pk + ks * C::kTileBytes + sl * slab, tail ? &tm_pk_tail : &tm_pk,
                                        bar(kBarKFull + ks), sl * 64, k * kBlockN, ph);
                    }
                    __syncwarp();
                    if (++ks == (uint32_t)p.stages) { ks = 0; kph ^= 1u; }
                }
                if (!ok) break;
            }
            if (SR) {
                // suffix K of the tile's candidates, block by block through the ring: one box of
                // Skv rows per candidate, candidates Spad rows apart inside a block
                const int nbs = items_of(t) - p.nblk_p;
#pragma unroll 1
                for (int j = 0; j < nbs; ++j) {
                    ok = mbar_wait_warp(bar(kBarKFree + ks), kph, abort_flag, p.status, kErrProducerK);
                    if (!ok) break;
                    if (long_sfx) {
                        // keys [128 j, 128 j + 128) of the tile's candidate; rows past the cache are zero-filled
                        if (elect_one_sync()) {
                            mbar_arrive_expect_tx(bar(kBarKFull + ks), (uint32_t)C::kTileBytes);
#pragma unroll 1
                            for (int sl = 0; sl < C::kSlabs; ++sl)
                                tma_load_4d(sbase + p.off_pk + ks * C::kTileBytes + sl * C::kSlabBytes, &tm_sk,
                                            bar(kBarKFull + ks), sl * 64, j * kBlockN, t.g, t.b_first);
                        }
                    } else {
                        const int ncb = sfx_block_cands(p, t.nc, j);
                        const int slab = sfx_block_rows(p, t.nc, j) * 128;
                        if (elect_one_sync()) {
                            mbar_arrive_expect_tx(bar(kBarKFull + ks), (uint32_t)(ncb * C::kSlabs * p.Skv * 128));
#pragma unroll 1
                            for (int c = 0; c < ncb; ++c)
#pragma unroll 1
                                for (int sl = 0; sl < C::kSlabs; ++sl)
                                    tma_load_4d(sbase + p.off_pk + ks * C::kTileBytes + sl * slab + c * p.Spad * 128,
                                                &tm_sk, bar(kBarKFull + ks), sl * 64, 0, t.g, t.b_first + j * p.cpb + c);
                        }
                    }
                    __syncwarp();
                    if (++ks == (uint32_t)p.stages) { ks = 0; kph ^= 1u; }
                }
                if (!ok) break;
            } else {
                // suffix K of the candidates this tile touches: one box per candidate
                if (elect_one_sync()) {
                    mbar_arrive_expect_tx(bar(kBarSKFull), (uint32_t)(t.nc * C::kSlabs * p.Sp * 128));
#pragma unroll 1
                    for (int c = 0; c < t.nc; ++c)
#pragma unroll 1
                        for (int sl = 0; sl < C::kSlabs; ++sl)
                            tma_load_4d(sbase + p.off_sk + sl * sfx_slab + c * p.Sp * 128, &tm_sk, bar(kBarSKFull),
                                        sl * 64, 0, t.g, t.b_first + c);
                }
                __syncwarp();
            }
            // Ask for the NEXT tile's Q in L2: its load can only be issued a tile from now, right when it is needed,
            // and then finds the data close by.  (Behind this tile's copies: the first ones of a launch are waited for.)
            if (tl + 1 < n_tiles) {
                const TileInfo tn = tile_info<MI == 2>(p, tile_at(tl + 1), t_begin);
                const int nseg_n = (SR && (!ANY || p.box.one_box)) ? 1 : p.fd_seg.div(tn.rows);
                int nb = p.fd_Rg.div(tn.R0), nr = tn.R0 - nb * p.Rg;
                if (elect_one_sync()) {
#pragma unroll 1
                    for (int s = 0; s < nseg_n; ++s) {
                        int c1, c2;
                        q_coords<ANY>(p, nr, tn.g, c1, c2);
#pragma unroll
                        for (int sl = 0; sl < C::kSlabs; ++sl) tma_prefetch_4d(&tm_q, sl * 64, c1, c2, nb);
                        nr += p.seg_rows;
                        if (nr >= p.Rg) {
                            nr -= p.Rg;
                            ++nb;
                        }
                    }
                }
                __syncwarp();
            }
        }
    } else if (role == 3) {
        // ------------------------------------------------------------------ producer, value side
        if (lane == 0) {
            prefetch_tensormap(&tm_sv);
            prefetch_tensormap(&tm_out);
            if (p.P > 0) { prefetch_tensormap(&tm_pv); prefetch_tensormap(&tm_pv_tail); }
        }
        // This warp also issues the TMA stores of each finished output tile.  The staging buffer
        // may share its shared memory with suffix V: tile t's output is staged after that tile's
        // last value MMA has read suffix V, and suffix V of tile t+1 is then fetched only once the
        // stores of tile t have read the staging buffer.
        const uint32_t stage = sbase + p.off_stage;
        uint32_t vs = 0, vph = 1;  // ring of V blocks: stage, parity of its release
        int store_slab = 0;  // slab_stage: slabs of the previous tile's output stored so far
        bool ok = true;
#pragma unroll 1
        for (int tl = 0; tl <= n_tiles && ok; ++tl) {
            const bool have_tile = tl < n_tiles;
            // Two jobs ride along with the prefix loads of tile tl: the stores of tile tl-1 (once it
            // is staged) and the fetch of this tile's suffix V (once its buffer is free: after those
            // stores when it doubles as the staging buffer, else after the previous tile's value MMAs).
            bool pend_store = tl > 0, pend_sv = have_tile && !SR;
            TileInfo t;
            int nk = 0;  // V blocks still to fetch through the ring for this tile
            int ph = 0;  // head index inside the prefix caches
            int kfirst = 0;
            if (have_tile) {
                t = tile_info<MI == 2>(p, tile_at(tl), t_begin);
                const int inst = inst_of(t);
                ph = inst * p.Hkv + t.g;
                kfirst = first_block(inst);
                if (RES) {
                    // the resident prefix V blocks are free once every value MMA of the previous tile
                    // has completed
                    ok = mbar_wait_warp(bar(kBarSVFree), (tl & 1) ^ 1, abort_flag, p.status, kErrProducerV);
                    if (!ok) break;
                    if (first_of_run(t, inst) && elect_one_sync()) {
#pragma unroll 1
                        for (int k = 0; k < p.nblk_p; ++k) {
                            const bool tail = k == p.nblk_p - 1;
                            const int slab = tail ? tail_slab : C::kSlabBytes;
                            mbar_arrive_expect_tx(bar(kBarVFull + k), (uint32_t)(C::kSlabs * slab));
#pragma unroll 1
                            for (int sl = 0; sl < C::kSlabs; ++sl)
                                tma_load_3d(sbase + p.off_pv + k * C::kTileBytes + sl * slab,
                                            tail ? &tm_pv_tail : &tm_pv, bar(kBarVFull + k), sl * 64, k * kBlockN, ph);
                        }
                    }
                    __syncwarp();
                } else {
                    nk = SR ? items_of(t) : p.nblk_p;
                }
            }
            int k = nk > 0 ? kfirst : 0;  // (nk stays 0 when the prefix is resident)
#pragma unroll 1
            while (ok && (k < nk || pend_store || pend_sv)) {
                const bool block = k >= nk;  // nothing else left to do for this tile: wait for the jobs
                if (k < nk) {
                    ok = mbar_wait_warp(bar(kBarVFree + vs), vph, abort_flag, p.status, kErrProducerV);
                    if (!ok) break;
                    if (SR && k >= p.nblk_p) {
                        // a suffix V block: one box of Skv rows per candidate, Spad rows apart
                        const int j = k - p.nblk_p;
                        if (long_sfx) {
                            if (elect_one_sync()) {
                                mbar_arrive_expect_tx(bar(kBarVFull + vs), (uint32_t)C::kTileBytes);
#pragma unroll 1
                                for (int sl = 0; sl < C::kSlabs; ++sl)
                                    tma_load_4d(sbase + p.off_pv + vs * C::kTileBytes + sl * C::kSlabBytes, &tm_sv,
                                                bar(kBarVFull + vs), sl * 64, j * kBlockN, t.g, t.b_first);
                            }
                        } else {
                            const int ncb = sfx_block_cands(p, t.nc, j);
                            const int slab = sfx_block_rows(p, t.nc, j) * 128;
                            if (elect_one_sync()) {
                                mbar_arrive_expect_tx(bar(kBarVFull + vs), (uint32_t)(ncb * C::kSlabs * p.Skv * 128));
#pragma unroll 1
                                for (int c = 0; c < ncb; ++c)
#pragma unroll 1
                                    for (int sl = 0; sl < C::kSlabs; ++sl)
                                        tma_load_4d(sbase + p.off_pv + vs * C::kTileBytes + sl * slab + c * p.Spad * 128,
                                                    &tm_sv, bar(kBarVFull + vs), sl * 64, 0, t.g,
                                                    t.b_first + j * p.cpb + c);
                            }
                        }
                    } else {
                        const bool tail = k == p.nblk_p - 1;
                        const int slab = tail ? tail_slab : C::kSlabBytes;
                        if (elect_one_sync()) {
                            mbar_arrive_expect_tx(bar(kBarVFull + vs), (uint32_t)(C::kSlabs * slab));
#pragma unroll 1
                            for (int sl = 0; sl < C::kSlabs; ++sl)
                                tma_load_3d(sbase + p.off_pv + vs * C::kTileBytes + sl * slab,
                                            tail ? &tm_pv_tail : &tm_pv, bar(kBarVFull + vs), sl * 64, k * kBlockN, ph);
                        }
                    }
                    __syncwarp();
                    if (++vs == (uint32_t)p.stages) { vs = 0; vph ^= 1u; }
                    ++k;
                }
                bool sv_ready = false;
                if (pend_sv && !alias_stage) {
                    if (tl == 0)
                        sv_ready = true;
                    else if (block)
                        sv_ready = ok = mbar_wait_warp(bar(kBarSVFree), (tl & 1) ^ 1, abort_flag, p.status, kErrProducerV);
                    else
                        sv_ready = __shfl_sync(0xffffffffu, mbar_try_wait(bar(kBarSVFree), (tl & 1) ^ 1) ? 1 : 0, 0) != 0;
                    if (!ok) break;
                }
                if (pend_store && !sv_ready) {
                    // the staging buffer holds the whole tile, or (slab_stage) one 64-column slab per round
                    const uint32_t round = slab_stage ? (uint32_t)((tl - 1) * C::kSlabs + store_slab) : (uint32_t)(tl - 1);
                    bool ready;
                    if (block)
                        ready = ok = mbar_wait_warp(bar(kBarStageFull), round & 1, abort_flag, p.status, kErrEpilogue);
                    else
                        ready = __shfl_sync(0xffffffffu, mbar_try_wait(bar(kBarStageFull), round & 1) ? 1 : 0, 0) != 0;
                    if (!ok) break;
                    if (ready) {
                        const TileInfo u = tile_info<MI == 2>(p, tile_at(tl - 1), t_begin);
                        const int nseg = (SR && (!ANY || p.box.one_box)) ? 1 : p.fd_seg.div(u.rows);
                        const int sl_first = slab_stage ? store_slab : 0;
                        const int sl_end = slab_stage ? store_slab + 1 : C::kSlabs;
                        if (elect_one_sync()) {
#pragma unroll 1
                            for (int sl = sl_first; sl < sl_end; ++sl)
#pragma unroll 1
                                for (int s = 0; s < nseg; ++s) {
                                    const int R = u.R0 + s * p.seg_rows;
                                    const int b = p.fd_Rg.div(R), r = R - b * p.Rg;
                                    if (PAD && r >= p.Rr) continue;  // padding only
                                    int c1, c2;
                                    q_coords<ANY>(p, r, u.g, c1, c2);
                                    tma_store_4d(&tm_out, stage + (slab_stage ? 0 : sl) * kStagingBytes + s * p.seg_rows * 128,
                                                 sl * 64, c1, c2, b);
                                }
                            tma_store_commit();
                            tma_store_wait_read();  // the staging buffer may be overwritten after this
                            mbar_arrive(bar(kBarStageFree));
                        }
                        __syncwarp();
                        PSKV_TRACE_EVENT(4, tl - 1);
                        if (slab_stage && store_slab + 1 < C::kSlabs) {
                            ++store_slab;
                        } else {
                            store_slab = 0;
                            pend_store = false;
                        }
                    }
                }
                if (pend_sv && alias_stage && !pend_store) sv_ready = true;
                if (sv_ready) {
                    if (elect_one_sync()) {
                        mbar_arrive_expect_tx(bar(kBarSVFull), (uint32_t)(t.nc * C::kSlabs * p.Sp * 128));
#pragma unroll 1
                        for (int c = 0; c < t.nc; ++c)
#pragma unroll 1
                            for (int sl = 0; sl < C::kSlabs; ++sl)
                                tma_load_4d(sbase + p.off_sv + sl * sfx_slab + c * p.Sp * 128, &tm_sv, bar(kBarSVFull),
                                            sl * 64, 0, t.g, t.b_first + c);
                    }
                    __syncwarp();
                    PSKV_TRACE_EVENT(5, tl);
                    pend_sv = false;
                }
            }
        }
        if (elect_one_sync()) tma_store_wait_all();
        __syncwarp();
    } else if (role == 1) {
        // ------------------------------------------------------------------ score MMAs: S = Q K^T
        // The two issuers.  An item is handed on as soon as its last MMA is issued, and the next one worked out behind that: working
        // it out in the middle of this one's MMAs delayed every item that somebody waits for, as in tiles of few items (1000 beams,
        // 32/32 heads, 2 tokens over 96 cached ones 303-318 us, now 296-302; 64 beams, P = 900, one over 120 19.1, now 18.6; 16 candidates, 32/8, P
        // = 256, S = 48 11.9, now 11.6), and 256 candidates, 32/8, P = 2048, S = 32 take 254 us instead of 262 too.  With rings the
        // positions are counters and the barriers are looked at together first, since as a rule everything is there (the last
        // shape by division and one barrier after another: 287).  With the prefix resident nearly every item is waited for, and the
        // compiler makes worse code of the counters (8 x 64 candidates, 32/8, P = 256, S = 48 172 us with them, else 153).  There the
        // order in which the two issuers' MMAs meet decides: working ahead took some calls from 203 to 187 us (509 candidates, 32/32,
        // P = 180, S = 38; 199 now) or 121 to 115 (150, P = 150, S = 96) and others from 94 to 99 (200, P = 200, S = 64; 97 now) or 57.5 to
        // 59.5 (300, 32/8, P = 200, S = 30), with no rule in the sizes; most lost.
        int tl = 0;
        uint32_t ks = 0, kph = 0;        // ring of K blocks: stage, parity of its loads
        uint32_t slot = 0, slot_ph = 1;  // score slot, parity of its release
        TileInfo t = tile_info<MI == 2>(p, tile_at(0), t_begin);
        int nitems = items_of(t);
        int kfirst = first_block(inst_of(t)), k = kfirst;
        const uint64_t q_desc = make_smem_desc(sbase + p.off_q, 0, 1024);
        bool ok = true;
#pragma unroll 1
        for (int i = 0; tl < n_tiles; ++i) {
            // everything that does not depend on a wait comes first, so that it is out of the way
            // when the waits return
            if (RES) {
                slot = (uint32_t)i % kSlots;
                slot_ph = (((uint32_t)i / kSlots) & 1u) ^ 1u;
            }
            uint32_t kaddr, kbar, kpar;
            int n, slab;
            bool kwait = true;
            if (k < p.nblk_p || SR) {
                n = k < p.nblk_p ? prefix_block_rows(p, k)
                    : long_sfx ? sfx_long_rows(p, k - p.nblk_p) : sfx_block_rows(p, t.nc, k - p.nblk_p);
                slab = (SR && long_sfx && k >= p.nblk_p) ? C::kSlabBytes : n * 128;  // (full 128-row boxes)
                if (RES) {
                    const int inst = inst_of(t);
                    kwait = first_of_run(t, inst);
                    kbar = bar(kBarKFull + k);
                    kpar = (uint32_t)(run_of(t, inst) - run_first) & 1u;
                    kaddr = sbase + p.off_pk + k * C::kTileBytes;
                } else {
                    kbar = bar(kBarKFull + ks);
                    kpar = kph;
                    kaddr = sbase + p.off_pk + ks * C::kTileBytes;
                }
            } else {
                n = t.n_sfx;
                slab = sfx_slab;
                kbar = bar(kBarSKFull);
                kpar = (uint32_t)tl & 1u;
                kaddr = sbase + p.off_sk;
            }
            const uint32_t idesc = make_idesc_bf16(kTileM, n, 0);
            const uint32_t d_tmem = tmem + slot * kBlockN;
            const uint64_t k_desc = make_smem_desc(kaddr, 0, 1024);
            const uint64_t k_slab = (uint64_t)(slab >> 4);
            const bool last_of_tile = k == nitems - 1;
            const bool free_stage = (k < p.nblk_p || SR) && !RES;
            // the slot is free once the value MMAs of item i-3 (which read P from it) have completed
            PSKV_TRACE_EVENT(16, i);
            const bool qwait = k == kfirst;
            bool ready = false;
            if (!RES) {
                ready = mbar_test_wait(bar(kBarPvDone + slot), slot_ph);
                if (kwait) ready &= mbar_test_wait(kbar, kpar);
                if (qwait) ready &= mbar_test_wait(bar(kBarQFull), tl & 1);
            }
            if (RES || !__all_sync(0xffffffffu, ready)) {
                ok = mbar_wait_warp(bar(kBarPvDone + slot), slot_ph, abort_flag, p.status, kErrMmaQk);
                PSKV_TRACE_EVENT(18, i);
                if (ok && qwait) ok = mbar_wait_warp(bar(kBarQFull), tl & 1, abort_flag, p.status, kErrMmaQk);
                if (ok && kwait) ok = mbar_wait_warp(kbar, kpar, abort_flag, p.status, kErrMmaQk);
                if (!ok) break;
            }
            if (MI && RES && k == kfirst && first_of_run(t, inst_of(t))) {
                // The resident copy of a run always loads every prefix block, also those this run skips as
                // padding.  Nobody multiplies them, so their loads are waited for here: a load must have
                // landed before its buffer and barrier are armed again for the next run, and before the
                // CTA exits.
                const uint32_t par = (uint32_t)(run_of(t, inst_of(t)) - run_first) & 1u;
                for (int kk = 0; kk < kfirst && kk < p.nblk_p && ok; ++kk)
                    ok = mbar_wait_warp(bar(kBarKFull + kk), par, abort_flag, p.status, kErrMmaQk);
                if (!ok) break;
            }
            PSKV_TRACE_EVENT(10, i);
            tc_fence_after();
            if (elect_one_sync()) {
#pragma unroll
                for (int ks16 = 0; ks16 < D / 16; ++ks16) {
                    const uint64_t qoff = (uint64_t)(((ks16 >> 2) * C::kSlabBytes + (ks16 & 3) * 32) >> 4);
                    const uint64_t koff = (uint64_t)(ks16 >> 2) * k_slab + (uint64_t)(((ks16 & 3) * 32) >> 4);
                    mma_ss(d_tmem, q_desc + qoff, k_desc + koff, idesc, ks16 > 0 ? 1u : 0u);
                }
                tc_commit(bar(kBarSFull + slot));
                if (free_stage) tc_commit(bar(kBarKFree + ks));
                if (last_of_tile) tc_commit(bar(kBarQkFree));  // the suffix block ends the tile's scores
            }
            __syncwarp();
            PSKV_TRACE_EVENT(12, i);
            if (free_stage && ++ks == (uint32_t)p.stages) { ks = 0; kph ^= 1u; }
            if (!RES && ++slot == kSlots) { slot = 0; slot_ph ^= 1u; }
            if (++k == nitems) {
                k = 0;
                if (++tl < n_tiles) {
                    t = tile_info<MI == 2>(p, tile_at(tl), t_begin);
                    nitems = items_of(t);
                    k = kfirst = first_block(inst_of(t));
                }
            }
        }
    } else if (role == 2) {
        // ------------------------------------------------------------------ value MMAs: O += P V
        int tl = 0;
        uint32_t vs = 0, vph = 0;        // ring of V blocks: stage, parity of its loads
        uint32_t slot = 0, slot_ph = 0;  // score slot, parity of its probabilities
        TileInfo t = tile_info<MI == 2>(p, tile_at(0), t_begin);
        int nitems = items_of(t);
        int kfirst = first_block(inst_of(t)), k = kfirst;
        const uint32_t idesc_pv = make_idesc_bf16(kTileM, D, 1);
        bool ok = true;
#pragma unroll 1
        for (int i = 0; tl < n_tiles; ++i) {
            // everything that does not depend on a wait comes first
            if (RES) {
                slot = (uint32_t)i % kSlots;
                slot_ph = ((uint32_t)i / kSlots) & 1u;
            }
            uint32_t vaddr, vbar, vpar;
            int n, slab;
            bool vwait = true;
            if (k < p.nblk_p || SR) {
                n = k < p.nblk_p ? prefix_block_rows(p, k)
                    : long_sfx ? sfx_long_rows(p, k - p.nblk_p) : sfx_block_rows(p, t.nc, k - p.nblk_p);
                slab = (SR && long_sfx && k >= p.nblk_p) ? C::kSlabBytes : n * 128;  // (full 128-row boxes)
                if (RES) {
                    const int inst = inst_of(t);
                    vwait = first_of_run(t, inst);
                    vbar = bar(kBarVFull + k);
                    vpar = (uint32_t)(run_of(t, inst) - run_first) & 1u;
                    vaddr = sbase + p.off_pv + k * C::kTileBytes;
                } else {
                    vbar = bar(kBarVFull + vs);
                    vpar = vph;
                    vaddr = sbase + p.off_pv + vs * C::kTileBytes;
                }
            } else {
                n = t.n_sfx;
                slab = sfx_slab;
                vbar = bar(kBarSVFull);
                vpar = (uint32_t)tl & 1u;
                vaddr = sbase + p.off_sv;
            }
            const uint32_t p_tmem = tmem + slot * kBlockN;  // bf16 pairs: 8 columns per 16 keys
            const uint64_t v_desc = make_smem_desc(vaddr, (uint32_t)slab, 1024);
            const int nk = n >> 4;
            const bool last_of_tile = k == nitems - 1;
            const bool free_stage = (k < p.nblk_p || SR) && !RES;
            const uint32_t acc0 = k > kfirst ? 1u : 0u;
            PSKV_TRACE_EVENT(17, i);
            const bool owait = k == kfirst && tl > 0;  // (O of the previous tile must have been read out by the epilogue warps)
            bool ready = false;
            if (!RES) {
                ready = mbar_test_wait(bar(kBarPReady + slot), slot_ph);
                if (vwait) ready &= mbar_test_wait(vbar, vpar);
                if (owait) ready &= mbar_test_wait(bar(kBarOFree), (tl - 1) & 1);
            }
            if (RES || !__all_sync(0xffffffffu, ready)) {
                ok = mbar_wait_warp(bar(kBarPReady + slot), slot_ph, abort_flag, p.status, kErrMmaPv);
                PSKV_TRACE_EVENT(15, i);
                if (ok && owait) ok = mbar_wait_warp(bar(kBarOFree), (tl - 1) & 1, abort_flag, p.status, kErrMmaPv);
                PSKV_TRACE_EVENT(14, i);
                if (ok && vwait) ok = mbar_wait_warp(vbar, vpar, abort_flag, p.status, kErrMmaPv);
                if (!ok) break;
            }
            if (MI && RES && k == kfirst && first_of_run(t, inst_of(t))) {  // (as for the K blocks above)
                const uint32_t par = (uint32_t)(run_of(t, inst_of(t)) - run_first) & 1u;
                for (int kk = 0; kk < kfirst && kk < p.nblk_p && ok; ++kk)
                    ok = mbar_wait_warp(bar(kBarVFull + kk), par, abort_flag, p.status, kErrMmaPv);
                if (!ok) break;
            }
            PSKV_TRACE_EVENT(11, i);
            tc_fence_after();
            if (elect_one_sync()) {
#pragma unroll
                for (int ks16 = 0; ks16 < kBlockN / 16; ++ks16) {
                    if (ks16 < nk) {
                        const uint32_t p_cols = p_tmem + (ks16 >> 1) * kPiece + (ks16 & 1) * 8;
                        const uint64_t v_rows = v_desc + (uint64_t)(ks16 * (2048 >> 4));
                        mma_ts(tmem + kOCol, p_cols, v_rows, idesc_pv, ks16 > 0 ? 1u : acc0);
                        if (TWO) mma_ts(tmem + kOCol, p_cols + kPiece / 2, v_rows, idesc_pv, 1u);
                    }
                }
                tc_commit(bar(kBarPvDone + slot));
                if (free_stage) tc_commit(bar(kBarVFree + vs));
                if (last_of_tile) {
                    tc_commit(bar(kBarSVFree));
                    tc_commit(bar(kBarOFull));
                }
            }
            __syncwarp();
            PSKV_TRACE_EVENT(13, i);
            if (free_stage && ++vs == (uint32_t)p.stages) { vs = 0; vph ^= 1u; }
            if (!RES && ++slot == kSlots) { slot = 0; slot_ph ^= 1u; }
            if (++k == nitems) {
                k = 0;
                if (++tl < n_tiles) {
                    t = tile_info<MI == 2>(p, tile_at(tl), t_begin);
                    nitems = items_of(t);
                    k = kfirst = first_block(inst_of(t));
                }
            }
        }
    } else if (warp < 4 + 4 * kGroups) {
        // ------------------------------------------------------------------ softmax warps (4..19)
        // Four warpgroups work on every item: the 128 score columns are four pieces of 32 and
        // group j takes piece j, so that each scheduler always has four independent softmax warps
        // to hide the others' tensor-memory and barrier latencies.  Each thread owns one query
        // row (tensor-memory lane): p = 2^(s * sl2), row sum, bf16 pairs written over the first
        // half of the piece they came from (a group only ever overwrites columns it has read
        // itself).  No running max is subtracted: bf16 and fp32 share an 8-bit exponent, so the
        // quotient O / l is exact to rounding for any row whose sum stays within [2^-100, 2^100];
        // a row outside that range (essentially never, it means logits beyond +-69 nats) is
        // redone with max subtraction by this CTA once its tiles are finished.  The groups share no
        // state; their partial row sums meet in the epilogue, which the same warps run for the
        // previous tile (group j normalises O columns [32j, 32j+32)) right after the first item
        // of the next one, when that tile's last value MMAs have long completed.
        const int wg = (warp - 4) >> 2;
        const int row = 32 * (warp & 3) + lane;
        const uint32_t lane_addr = (uint32_t)(32 * (warp & 3)) << 16;
        bool ok = true;
        float lsum = 0.f;
        int item = 0;  // items handled so far
#pragma unroll 1
        for (int tl = 0; tl < n_tiles && ok; ++tl) {
            const TileInfo t = tile_info<MI == 2>(p, tile_at(tl), t_begin);
            const int nitems = items_of(t);
            int lo_sfx = 1, hi_sfx = 0;
            int k_own = p.nblk_p;  // suffix-ring mode: the item that holds this row's candidate
            if (row < t.rows) {
                const int R = t.R0 + row;
                const int b = p.fd_Rg.div(R), r = R - b * p.Rg;
                const int i = r - p.fd_S.div(r) * Sh;  // query index inside the candidate
                if ((PAD && r >= p.Rr) || (ANY && i >= p.S)) {
                    // a padding row between two candidates: sees no suffix key, is never stored
                } else if (SR) {
                    // query i is suffix token L - S + i of its candidate: suffix keys 0 .. L - S + i
                    const int pos = suffix_tokens(p.suffix_len, b, p.S, p.Skv) - p.S + i;
                    if (long_sfx) {
                        lo_sfx = 0;
                        hi_sfx = pos;  // counted from the candidate's first key; block j starts at 128 j
                    } else {
                        const int c = b - t.b_first, j = p.fd_cpb.div(c);
                        k_own += j;
                        lo_sfx = (c - j * p.cpb) * p.Spad;
                        hi_sfx = lo_sfx + pos;
                    }
                } else {
                    lo_sfx = (b - t.b_first) * p.Sp;  // first suffix column of this row's candidate
                    hi_sfx = lo_sfx + i;              // causal: suffix keys 0..i
                }
            }
            lsum = 0.f;
            // several instructions: the first `pad` prefix keys of this tile's instruction are left padding
            const int pad = MI ? p.pad[inst_of(t)] : 0;
#pragma unroll 1
            for (int k = pad / kBlockN; k < nitems && ok; ++k, ++item) {
                {
                    const int slot = item % kSlots;
                    const uint32_t s_tmem = tmem + lane_addr + slot * kBlockN + wg * kPiece;
                    // valid columns of this row: [lo, hi].  Padding rows of a tile take part in prefix
                    // blocks like real rows and see no suffix key.  They are never stored; where no copy wrote
                    // them their scores are whatever shared memory held, NaN included, and the epilogue stages
                    // zeros for such rows.
                    int n, lo, hi;
                    if (k < p.nblk_p) {
                        n = prefix_block_rows(p, k);
                        lo = max(0, pad - k * kBlockN);
                        hi = min(kBlockN, p.P - k * kBlockN) - 1;
                    } else if (SR && long_sfx) {
                        n = sfx_long_rows(p, k - p.nblk_p);
                        lo = lo_sfx;  // 0 for a real row, 1 (with hi 0 - ...: nothing visible) for padding
                        hi = lo_sfx == 0 ? hi_sfx - (k - p.nblk_p) * kBlockN : 0;
                    } else if (SR) {
                        n = sfx_block_rows(p, t.nc, k - p.nblk_p);
                        lo = k == k_own ? lo_sfx : 1;  // other candidates' blocks: nothing visible
                        hi = k == k_own ? hi_sfx : 0;
                    } else {
                        n = t.n_sfx;
                        lo = lo_sfx;
                        hi = hi_sfx;
                    }
                    const int c0 = wg * kPiece;  // first column of my piece
                    // my piece: 0 = not read by the value MMAs, 1 = no valid column for this warp
                    // (zeros), 2 = some columns masked, 3 = all columns valid for all rows
                    int kind = 0;
                    if (c0 < n) {
                        const bool all_valid = lo <= c0 && hi >= c0 + kPiece - 1;
                        const bool none_valid = hi < lo || hi < c0 || lo > c0 + kPiece - 1;
                        kind = __all_sync(0xffffffffu, all_valid) ? 3 : __all_sync(0xffffffffu, none_valid) ? 1 : 2;
                    }
                    PSKV_TRACE_EVENT(25, item);
                    ok = mbar_wait_warp(bar(kBarSFull + slot), (item / kSlots) & 1, abort_flag, p.status, kErrSoftmax);
                    if (!ok) break;
                    tc_fence_after();
                    PSKV_TRACE_EVENT(20, item);
                    if (kind != 0) {
                        uint32_t rr[kPiece], pk[kPiece / 2];
                        if (kind >= 2) {
                            tmem_ld32(s_tmem, rr);
                            tmem_wait_ld();
                        }
                        PSKV_TRACE_EVENT(21, item);
                        float ls0 = 0.f, ls1 = 0.f;
                        if (kind >= 2) {
                            // all exponentials first (independent, so they pipeline through the
                            // special-function unit), then sums and bf16 pairs
                            float e[kPiece];
#pragma unroll
                            for (int c = 0; c < kPiece; c += 2) {
                                float x0 = __uint_as_float(rr[c]), x1 = __uint_as_float(rr[c + 1]);
                                mul_f32x2(x0, x1, p.sl2);
                                e[c] = ex2_approx(x0);
                                e[c + 1] = ex2_approx(x1);
                            }
                            if (kind == 2) {
                                const unsigned span = (unsigned)(hi - lo);
                                const int base = c0 - lo;
                                const bool any_col = hi >= lo;
#pragma unroll
                                for (int c = 0; c < kPiece; ++c)
                                    e[c] = (any_col && (unsigned)(base + c) <= span) ? e[c] : 0.f;
                            }
                            float ls2 = 0.f, ls3 = 0.f;
#pragma unroll
                            for (int c = 0; c < kPiece / 4; ++c) {
                                add_f32x2(ls0, ls1, e[4 * c], e[4 * c + 1]);
                                add_f32x2(ls2, ls3, e[4 * c + 2], e[4 * c + 3]);
                                pk[2 * c] = pack_bf16x2(e[4 * c], e[4 * c + 1]);
                                pk[2 * c + 1] = pack_bf16x2(e[4 * c + 2], e[4 * c + 3]);
                            }
                            if (TWO) {  // what the rounding leaves is exact in fp32
                                uint32_t lo[kPiece / 2];
#pragma unroll
                                for (int c = 0; c < kPiece / 2; ++c)
                                    lo[c] = pack_bf16x2(e[2 * c] - __uint_as_float(pk[c] << 16), e[2 * c + 1] - __uint_as_float(pk[c] & 0xffff0000u));
                                tmem_st16(s_tmem + kPiece / 2, lo);
                            }
                            ls0 += ls2;
                            ls1 += ls3;
                        } else {
#pragma unroll
                            for (int c = 0; c < kPiece / 2; ++c) pk[c] = 0u;
                            if (TWO) tmem_st16(s_tmem + kPiece / 2, pk);
                        }
                        lsum += ls0 + ls1;
                        tmem_st16(s_tmem, pk);
                    }
                    if (k == nitems - 1) {
                        // the tile's partial row sums go to the epilogue warps through shared memory (kept
                        // for four tiles, or for one: then the epilogue must have read the previous tile's)
                        if (p.ml_mask == 0 && tl > 0) {
                            ok = mbar_wait_warp(bar(kBarMlFree), (tl - 1) & 1, abort_flag, p.status, kErrSoftmax);
                            if (!ok) break;
                        }
                        ml[((tl & p.ml_mask) * kGroups + wg) * kTileM + row] = lsum;
                        __threadfence_block();
                    }
                    PSKV_TRACE_EVENT(23, item);
                    tmem_wait_st();
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(bar(kBarPReady + slot));
                    PSKV_TRACE_EVENT(24, item);
                }
            }
        }
    } else {
        // ------------------------------------------------------------------ epilogue warps (20..23)
        // O / l -> bf16 -> staging buffer (TMA-stored by warp 3); lse; rows to redo.  Thread <->
        // query row; the row sum is the sum of the four softmax groups' partial sums.
        const int ew = warp & 3;
        const int row = 32 * ew + lane;
        const uint32_t lane_addr = (uint32_t)(32 * ew) << 16;
        bool ok = true;
#pragma unroll 1
        for (int te = 0; te < n_tiles && ok; ++te) {
            const TileInfo u = tile_info<MI == 2>(p, tile_at(te), t_begin);
            ok = mbar_wait_warp(bar(kBarOFull), te & 1, abort_flag, p.status, kErrEpilogue);
            if (!ok) break;
            PSKV_TRACE_EVENT(30, te);
            tc_fence_after();
            const float *mlt = ml + (te & p.ml_mask) * kGroups * kTileM + row;
            const float l = (mlt[0] + mlt[kTileM]) + (mlt[2 * kTileM] + mlt[3 * kTileM]);
            __syncwarp();
            if (lane == 0) mbar_arrive(bar(kBarMlFree));
            const bool row_ok = l >= kMinRowSum && l <= kMaxRowSum;  // false for overflow (inf, NaN), underflow
            // staged values must be finite (the buffer may double as suffix V, whose padding rows
            // meet zero probabilities): rows that failed stage zeros and are redone, and so do padding rows, whose
            // sums may be NaN (they are not redone)
            const float inv = row_ok ? 1.f / l : 0.f;
            if (slab_stage) {
                // One 64-column slab at a time through a staging buffer of one slab: load, hand O back after
                // the last load, wait for the previous slab's stores to have read the buffer, stage, tell
                // the storing warp.  The buffer is this kernel's own: suffix V of the next tile is fetched
                // as soon as this tile's value MMAs have completed, not behind these stores.
#pragma unroll 1
                for (int sl = 0; sl < C::kSlabs; ++sl) {
                    const uint32_t round = (uint32_t)(te * C::kSlabs + sl);
                    uint32_t o0[kPiece], o1[kPiece];
                    tmem_ld32(tmem + lane_addr + kOCol + sl * 64, o0);
                    tmem_ld32(tmem + lane_addr + kOCol + sl * 64 + kPiece, o1);
                    tmem_wait_ld();
                    PSKV_TRACE_EVENT(34 + sl, te);
                    if (sl == C::kSlabs - 1) {
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(bar(kBarOFree));
                        PSKV_TRACE_EVENT(32, te);
                    }
                    ok = mbar_wait_warp(bar(kBarStageFree), (round & 1) ^ 1, abort_flag, p.status, kErrEpilogue);
                    if (!ok) break;
                    uint8_t *srow = smem + p.off_stage + row * 128;
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        uint4 v;
                        v.x = pack_bf16x2(__uint_as_float(o0[8 * c]) * inv, __uint_as_float(o0[8 * c + 1]) * inv);
                        v.y = pack_bf16x2(__uint_as_float(o0[8 * c + 2]) * inv, __uint_as_float(o0[8 * c + 3]) * inv);
                        v.z = pack_bf16x2(__uint_as_float(o0[8 * c + 4]) * inv, __uint_as_float(o0[8 * c + 5]) * inv);
                        v.w = pack_bf16x2(__uint_as_float(o0[8 * c + 6]) * inv, __uint_as_float(o0[8 * c + 7]) * inv);
                        if (!row_ok) v = make_uint4(0, 0, 0, 0);
                        *reinterpret_cast<uint4 *>(srow + ((c ^ (row & 7)) << 4)) = v;
                    }
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        uint4 v;
                        v.x = pack_bf16x2(__uint_as_float(o1[8 * c]) * inv, __uint_as_float(o1[8 * c + 1]) * inv);
                        v.y = pack_bf16x2(__uint_as_float(o1[8 * c + 2]) * inv, __uint_as_float(o1[8 * c + 3]) * inv);
                        v.z = pack_bf16x2(__uint_as_float(o1[8 * c + 4]) * inv, __uint_as_float(o1[8 * c + 5]) * inv);
                        v.w = pack_bf16x2(__uint_as_float(o1[8 * c + 6]) * inv, __uint_as_float(o1[8 * c + 7]) * inv);
                        if (!row_ok) v = make_uint4(0, 0, 0, 0);
                        *reinterpret_cast<uint4 *>(srow + (((4 + c) ^ (row & 7)) << 4)) = v;
                    }
                    fence_proxy_async();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(bar(kBarStageFull));
                }
                if (!ok) break;
            } else {
            // the TMA stores of the previous tile must have read the staging buffer
                ok = mbar_wait_warp(bar(kBarStageFree), (te & 1) ^ 1, abort_flag, p.status, kErrEpilogue);
                if (!ok) break;
                PSKV_TRACE_EVENT(33, te);
                // one 64-column slab per round; O is free for the next tile's first value MMA as soon
                // as the last round's loads have returned
    #pragma unroll 1
                for (int sl = 0; sl < C::kSlabs; ++sl) {
                    uint32_t o0[kPiece], o1[kPiece];
                    tmem_ld32(tmem + lane_addr + kOCol + sl * 64, o0);
                    tmem_ld32(tmem + lane_addr + kOCol + sl * 64 + kPiece, o1);
                    tmem_wait_ld();
                    PSKV_TRACE_EVENT(34 + sl, te);
                    if (sl == C::kSlabs - 1) {
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(bar(kBarOFree));
                        PSKV_TRACE_EVENT(32, te);
                    }
                    // 128-byte rows, 16-byte chunks swizzled by the row
                    uint8_t *srow = smem + p.off_stage + sl * kStagingBytes + row * 128;
    #pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        uint4 v;
                        v.x = pack_bf16x2(__uint_as_float(o0[8 * c]) * inv, __uint_as_float(o0[8 * c + 1]) * inv);
                        v.y = pack_bf16x2(__uint_as_float(o0[8 * c + 2]) * inv, __uint_as_float(o0[8 * c + 3]) * inv);
                        v.z = pack_bf16x2(__uint_as_float(o0[8 * c + 4]) * inv, __uint_as_float(o0[8 * c + 5]) * inv);
                        v.w = pack_bf16x2(__uint_as_float(o0[8 * c + 6]) * inv, __uint_as_float(o0[8 * c + 7]) * inv);
                        if (!row_ok) v = make_uint4(0, 0, 0, 0);  // (inf or NaN accumulators times zero are not zero)
                        *reinterpret_cast<uint4 *>(srow + ((c ^ (row & 7)) << 4)) = v;
                    }
    #pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        uint4 v;
                        v.x = pack_bf16x2(__uint_as_float(o1[8 * c]) * inv, __uint_as_float(o1[8 * c + 1]) * inv);
                        v.y = pack_bf16x2(__uint_as_float(o1[8 * c + 2]) * inv, __uint_as_float(o1[8 * c + 3]) * inv);
                        v.z = pack_bf16x2(__uint_as_float(o1[8 * c + 4]) * inv, __uint_as_float(o1[8 * c + 5]) * inv);
                        v.w = pack_bf16x2(__uint_as_float(o1[8 * c + 6]) * inv, __uint_as_float(o1[8 * c + 7]) * inv);
                        if (!row_ok) v = make_uint4(0, 0, 0, 0);
                        *reinterpret_cast<uint4 *>(srow + (((4 + c) ^ (row & 7)) << 4)) = v;
                    }
                }
                fence_proxy_async();
                __syncwarp();
                if (lane == 0) mbar_arrive(bar(kBarStageFull));
            }
            const int R = u.R0 + row;
            const int b = p.fd_Rg.div(R), r = R - b * p.Rg;
            const int hd = ANY ? p.fd_S.div(r) : 0, skip = ANY ? hd * (p.box.Sh - p.S) : 0;  // (head_box: padding rows before this head)
            const bool stored = row < u.rows && (!PAD || r < p.Rr) && (!ANY || r - hd * p.box.Sh < p.S);
            if (stored) {
                const size_t grow = ((size_t)b * p.Hq + (size_t)u.g * p.n_rep) * p.S + r - skip;
                // (log2f is good to 2^-22 absolute, more than the CUDA-core kernel loses, whose sum is relative to the maximum)
                p.lse[grow] = row_ok ? (TWO ? (float)log((double)l) : log2f(l) * kLn2) : __int_as_float(0x7fc00000);
            }
            const unsigned bad = __ballot_sync(0xffffffffu, stored && !row_ok);
            if (bad != 0u && lane == 0) atomicAdd(cta_redo, __popc(bad));
            PSKV_TRACE_EVENT(31, te);
        }
    }

    // ---------------------------------------------------------------------- teardown
    PSKV_TRACE_FLUSH;
    if (*abort_flag != 0) __nanosleep(20000);  // let copies and MMAs still in flight drain
    tc_fence_before();
    __syncthreads();
    if (warp == 2) tmem_dealloc(tmem, 512);
    // Rows whose sum left the safe range carry a NaN lse (and zeros in `out`): all warps of the CTA
    // now walk over its tiles and recompute those rows one warp per row with a running maximum.
    // Every role has finished, the stores of `out` have completed, so the data area of shared
    // memory is free: each warp stages its query row there.
    if (*cta_redo > 0 && *abort_flag == 0) {
        float *q_s = reinterpret_cast<float *>(smem) + warp * D;
#pragma unroll 1
        for (int tl = 0; tl < n_tiles; ++tl) {
            const TileInfo t = tile_info<MI == 2>(p, tile_at(tl), t_begin);
#pragma unroll 1
            for (int r = warp; r < t.rows; r += kThreads / 32) {
                const int R = t.R0 + r;
                const int b = p.fd_Rg.div(R), rr = R - b * p.Rg;
                const int hd = ANY ? p.fd_S.div(rr) : 0;
                if ((PAD && rr >= p.Rr) || (ANY && rr - hd * p.box.Sh >= p.S)) continue;
                const long long grow = ((long long)b * p.Hq + (long long)t.g * p.n_rep) * p.S + rr - (ANY ? hd * (p.box.Sh - p.S) : 0);
                const float v = p.lse[grow];
                if (v != v) {
                    if (MI) {  // the row's own prefix cache, without its left padding
                        const int inst = inst_of(t), pd = p.pad[inst];
                        FwdArgs a2 = p.args;
                        const size_t off = ((size_t)inst * p.Hkv * p.P + (size_t)pd) * D;
                        a2.prefix_k += off;
                        a2.prefix_v += off;
                        a2.dims.P = p.P - pd;
                        fwd_row<D>(a2, grow, q_s, lane);
                    } else {
                        fwd_row<D>(p.args, grow, q_s, lane);
                    }
                }
            }
        }
    }
}

// ------------------------------------------------------------------------------ host side

struct TilePlan {
    bool ok;
    int mode;   // kernel template MODE: 0 rings, 1 resident prefix, 2 / 3 suffix-ring (see there)
    int cbox, Spad, cpb;  // suffix-ring mode: candidates per tile, rows per candidate in a block, candidates per block
    int long_sfx;         // suffix-ring mode: tiles inside one candidate, its suffix keys in 128-key blocks
    int two_terms;        // suffix-ring mode: probabilities as two bf16 terms
    int tile_rows, seg_rows, tiles_per_group, sfx_rows;
    int Rp, Sp;           // rows / suffix key columns a candidate takes
    int Sh, one_box, head_box;  // see TcFwdParams
    double cost;          // estimated SM cycles of a KV head's tiles
    int nblk_p, tail_rows, resident, stages, alias_stage, slab_stage, ml_tiles;
    int off_pk, off_pv, off_q, off_sk, off_sv, off_stage, off_bar, off_misc, off_ml, smem_bytes;
};

// Cycles of a tile, for the choice of a tiling: about 2 000 per key block, 1 700 for the tile itself, and 100 per
// 64-column slab of a box of Q and of `out`: one thread asks for the next tile's boxes, fetches and stores them, and the single Q
// buffer is waited for (448 tiles of one box, 28 candidates, 32/8 heads, P = 190, S = 61, 15.8 us; 440 of sixteen 17.2; 262
// candidates, 4/4 heads, P = 20, S = 8 8.3 us in 68 tiles of sixteen boxes, 6.7 in 132 of eight).
double tile_cost(double blocks, double slabs) { return 2000.0 * blocks + 1700.0 + 100.0 * slabs; }

// Rows a candidate takes in the row list (Rp >= n_rep * S) and rows per tile, both multiples of 8, such that the
// suffix keys of all candidates a tile can touch (Sp columns each) fit one 128-key block.  Suffix lengths are
// rarely multiples of anything, so a candidate's rows are padded: by as much as makes the launch cheapest,
// which is more than to the next multiple of 8 where that lets a tile be fetched in few boxes
// (4 heads x 53 rows: 224 rows, 32-row boxes) or end where a candidate ends (4 x 113: 480 rows, tiles of 120).
// Measured against the suffix-ring tiling that took every length that is no multiple of 8 (whole calls):
// B = 333, 32/8 heads, P = 217, S = 53 173 -> 120 us; B = 64, 32/32, P = 230, S = 85 74 -> 57; B = 42, 32/8, P = 112,
// S = 117 44 -> 36; and against tiles of the largest divisor: B = 128, 32/8, P = 256, S = 80 (336 rows, three tiles
// of 112, instead of four of 80) 101 -> 82.
//
// ring: the suffix keys come in several blocks through the K / V rings, so a tile may touch any number of candidates.
// several: tiles for several instructions in one launch, where an instruction had better be whole tiles: the sum over all
// tiles decides, and boxes count less.
bool pick_tile_rows(const Dims &dm, bool ring, bool several, TilePlan *pl, int *nc_max)
{
    const int Sp = round_up(dm.S, 8);
    if (Sp > kBlockN) return false;
    const int Rg = dm.n_rep * dm.S, nblk = (dm.P + kBlockN - 1) / kBlockN, cpb = kBlockN / Sp;
    // The busiest SM's tiles decide, and among equals the sum over all: 133 candidates of 7 heads x 40 rows are 291 tiles of 128
    // rows in sixteen boxes or 333 of 112 in seven, which is cheaper in sum, but three rounds of the SMs instead of two.
    const long long sms = sm_count();
    const double slabs = several ? 0.6 : dm.d / 64;  // of a box
    auto score = [&](long long tiles, double cycles) {
        const long long all = tiles * dm.Hkv;
        if (several) return (double)tiles * cycles;
        return ((double)((all + sms - 1) / sms) + 0.25 * (double)all / (double)sms) * cycles;
    };
    double best = -1.0;
    for (int Rp = round_up(Rg, 8); Rp < Rg + kTileM; Rp += 8) {
        if ((long long)dm.B * Rp > 2000000000ll) break;
        if (best >= 0.0 && score(((long long)dm.B * Rp + kTileM - 1) / kTileM, tile_cost(nblk + 1, slabs)) >= best) break;
        for (int m = kTileM; m >= 8; m -= 8) {
            const int seg = gcd_int(Rp, m);
            // candidates that a window of m rows can touch, its offset in a candidate being a multiple of seg
            int nc = m % Rp == 0 ? m / Rp : Rp % m == 0 ? 1 : (m - seg + Rp - 1) / Rp + 1;
            if (nc > dm.B) nc = dm.B;
            if (!ring && nc * Sp > kBlockN) continue;
            const long long tiles = ((long long)dm.B * Rp + m - 1) / m;
            // suffix blocks of a tile: one, or (ring) one and a share for each candidate it touches beyond the first
            const double sfx = ring ? 1.0 + (double)(m - seg) / Rp / cpb : 1.0;
            const double cycles = tile_cost(nblk + sfx, slabs * (m / seg)), sc = score(tiles, cycles);
            if (best < 0.0 || sc < best) {
                best = sc;
                pl->cost = (double)tiles * cycles;
                pl->Rp = Rp;
                pl->tile_rows = m;
                pl->seg_rows = seg;
                pl->tiles_per_group = (int)tiles;
                *nc_max = nc;
            }
        }
    }
    if (best < 0.0) return false;
    pl->Sp = Sp;
    return true;
}

// Shared memory of the suffix-ring mode: K and V rings, Q, the staging buffer.
void layout_ring(const Dims &dm, TilePlan *pl)
{
    pl->nblk_p = (dm.P + kBlockN - 1) / kBlockN;
    pl->tail_rows = pl->nblk_p ? round_up(dm.P - (pl->nblk_p - 1) * kBlockN, 16) : 0;
    const int slabs = dm.d / 64;
    const int tile_bytes = slabs * kTileM * 128;
    const int ml_bytes = 4 * kGroups * kTileM * 4;
    const int stage_bytes = slabs * kStagingBytes;
    const int fixed = tile_bytes /*Q*/ + stage_bytes + ml_bytes + 64 + kBarBytes;
    int st = (kMaxSmem - fixed) / (2 * tile_bytes);
    if (st > kMaxStages) st = kMaxStages;
    if (st < 1) return;
    pl->stages = st;
    pl->off_pk = 0;
    pl->off_pv = st * tile_bytes;
    pl->off_q = 2 * st * tile_bytes;
    pl->off_sk = pl->off_sv = pl->off_stage = pl->off_q + tile_bytes;  // no suffix buffers of their own
    pl->off_bar = pl->off_stage + stage_bytes;
    pl->off_misc = pl->off_bar + kBarBytes;
    pl->off_ml = pl->off_misc + 64;
    pl->smem_bytes = pl->off_ml + ml_bytes;
    pl->ok = pl->smem_bytes <= kMaxSmem;
}

// Suffix-ring mode: a tile is the largest run of whole candidates with at most 128 rows; the
// suffix keys follow the prefix blocks through K/V rings, 128 / Spad candidates per block.
TilePlan plan_suffix_ring(const Dims &dm)
{
    TilePlan pl;
    memset(&pl, 0, sizeof(pl));
    const int Rg = dm.n_rep * dm.S;
    pl.mode = 2;
    if (Rg > kTileM || dm.Skv > kBlockN) {
        // Long suffixes: a tile lies inside one candidate, whose suffix keys come in blocks of 128.  Beyond 128 queries
        // it lies inside one head too: a head's rows are padded to whole tiles, so any length does, and a tile's
        // cost follows from its position, so that tiles can be dealt out by cost.  Else, and where heads would be
        // padded to more tiles, a tile is the largest divisor of the candidate's rows that fits.  (Lengths without such a
        // divisor went to the CUDA-core kernel: 1.58 ms for a prompt of 1039 tokens, 12.2 for 3001, now 24 and 108 us;
        // they keep its precision, see TWO at the kernel.)
        int rows = 0;
        for (int m = kTileM; m >= 16 && !rows; --m)
            if (Rg % m == 0) rows = m;
        if (!rows && Rg <= kTileM) rows = Rg;
        pl.two_terms = !rows;
        const int per_head = (dm.S + kTileM - 1) / kTileM;
        const long long head_tiles = (long long)dm.n_rep * per_head;
        if (dm.S > kTileM && (!rows || head_tiles < Rg / rows || (head_tiles == Rg / rows && dm.S % rows != 0))) {
            rows = round_up((dm.S + per_head - 1) / per_head, 8);
            if (dm.S % rows != 0) {
                pl.mode = 3;
                pl.head_box = 1;
                pl.Sh = rows * per_head;
            }
        }
        if (!rows) return pl;  // no usable divisor: the general kernels take the shape
        pl.Rp = pl.head_box ? dm.n_rep * pl.Sh : Rg;
        pl.one_box = 1;
        if ((long long)dm.B * pl.Rp > 2000000000ll) return pl;
        pl.long_sfx = 1;
        pl.Spad = 8;
        pl.cpb = 1;
        pl.cbox = 1;
        pl.tile_rows = pl.seg_rows = rows;
        pl.tiles_per_group = dm.B * (pl.Rp / rows);
    } else {
        pl.Spad = round_up(dm.Skv, 8);
        pl.cpb = kBlockN / pl.Spad;
        const int cmax = kTileM / Rg < dm.B ? kTileM / Rg : dm.B;
        // Candidates per tile: as many as fit, unless fewer give more SMs a tile or make a round less: a CTA's time is
        // its tiles times the key blocks of a tile, and the suffix blocks of a tile grow with its candidates.  With 512
        // candidates of one query row x 4 heads, 32 per tile are 128 tiles of 18 blocks on 148 SMs, 30 per tile
        // are 144 tiles of 17; 24 candidates with 126 cached tokens are 8 tiles of 28 blocks, or 96 of 6 (25 -> 13 us; 40
        // candidates of 64 tokens on 32/32 heads 27 -> 16; 131 with a prefix of 1872 28 -> 24).
        const int sms = sm_count();
        const int nblk = (dm.P + kBlockN - 1) / kBlockN;
        long long best_cost = -1;
        pl.cbox = cmax;
        for (int c = cmax; c >= 1; --c) {
            const long long tiles = (long long)dm.Hkv * ((dm.B + c - 1) / c);
            const long long rounds = (tiles + sms - 1) / sms;
            const long long cost = rounds * (nblk + (c + pl.cpb - 1) / pl.cpb + 1);
            if (best_cost < 0 || cost < best_cost) {
                best_cost = cost;
                pl.cbox = c;
            }
        }
        pl.mode = 3;
        pl.Rp = Rg;
        pl.one_box = 1;
        pl.tile_rows = pl.seg_rows = Rg * pl.cbox;
        pl.tiles_per_group = (dm.B + pl.cbox - 1) / pl.cbox;
        pl.cost = (double)pl.tiles_per_group * tile_cost(nblk + (pl.cbox + pl.cpb - 1) / pl.cpb, dm.d / 64);
    }
    layout_ring(dm, &pl);
    return pl;
}

// Lays out shared memory: all prefix blocks of a KV head if they fit beside the other buffers (resident mode), else
// rings of 2..4 block stages.
TilePlan plan_base(const Dims &dm, bool several)
{
    TilePlan pl;
    memset(&pl, 0, sizeof(pl));
    int nc_best = 0;
    if (!pick_tile_rows(dm, false, several, &pl, &nc_best)) return pl;
    pl.sfx_rows = round_up(nc_best * pl.Sp, 16);
    pl.nblk_p = (dm.P + kBlockN - 1) / kBlockN;
    pl.tail_rows = pl.nblk_p ? round_up(dm.P - (pl.nblk_p - 1) * kBlockN, 16) : 0;

    const int slabs = dm.d / 64;
    const int tile_bytes = slabs * kTileM * 128;
    const int sfx_bytes = round_up(slabs * pl.sfx_rows * 128, 1024);
    const int tail_bytes = round_up(slabs * pl.tail_rows * 128, 1024);
    const int ml_bytes = 4 * kGroups * kTileM * 4;  // partial row sums of four tiles in flight
    const int stage_bytes = slabs * kStagingBytes;
    const int tail_area = ml_bytes + 64 /*misc*/ + kBarBytes;
    // The output staging buffer gets memory of its own when that costs neither the residency of
    // the prefix nor a ring stage; otherwise it shares the suffix V buffer (value-side producer).
    const int fixed_own = tile_bytes /*Q*/ + 2 * sfx_bytes + stage_bytes + tail_area;
    const int shared_sv = sfx_bytes > stage_bytes ? sfx_bytes : stage_bytes;
    const int fixed_shared = tile_bytes + sfx_bytes + shared_sv + tail_area;
    const int resident_bytes = pl.nblk_p ? (pl.nblk_p - 1) * tile_bytes + tail_bytes : 0;
    auto ring_stages = [&](int fixed) {
        const int st = (kMaxSmem - fixed) / (2 * tile_bytes);
        return st > kMaxStages ? kMaxStages : st;
    };
    int kv_bytes = 0;  // bytes of the prefix K area (the V area has the same size)
    if (pl.nblk_p <= kMaxStages && fixed_shared + 2 * resident_bytes <= kMaxSmem) {
        pl.resident = 1;
        pl.stages = pl.nblk_p;
        kv_bytes = resident_bytes;
        pl.alias_stage = fixed_own + 2 * resident_bytes <= kMaxSmem ? 0 : 1;
        // Sharing the staging buffer with suffix V chains the next tile's suffix V behind this tile's
        // stores.  A staging buffer of one 64-column slab, with the partial row sums kept for one tile
        // instead of four, may still fit beside everything else: then the output goes a slab at a time.
        const int ml_one = kGroups * kTileM * 4;
        const int fixed_slab = tile_bytes + 2 * sfx_bytes + kStagingBytes + ml_one + 64 + kBarBytes;
        if (pl.alias_stage && slabs == 2 && fixed_slab + 2 * resident_bytes <= kMaxSmem) {
            pl.alias_stage = 0;
            pl.slab_stage = 1;
            pl.ml_tiles = 1;
        }
    } else {
        const int st = ring_stages(fixed_shared);
        if (st < 1) return pl;  // does not fit: the general kernels take the shape
        pl.stages = st;
        kv_bytes = st * tile_bytes;
        pl.alias_stage = ring_stages(fixed_own) == st ? 0 : 1;
    }
    const int sv_bytes = pl.alias_stage ? shared_sv : sfx_bytes;
    pl.off_pk = 0;
    pl.off_pv = pl.off_pk + kv_bytes;
    pl.off_q = pl.off_pv + kv_bytes;
    pl.off_sk = pl.off_q + tile_bytes;
    pl.off_sv = pl.off_sk + sfx_bytes;
    pl.off_stage = pl.alias_stage ? pl.off_sv : pl.off_sv + sv_bytes;
    pl.off_bar = pl.off_stage + (pl.alias_stage ? sv_bytes : pl.slab_stage ? kStagingBytes : stage_bytes);
    pl.off_misc = pl.off_bar + kBarBytes;
    pl.off_ml = pl.off_misc + 64;
    pl.smem_bytes = pl.off_ml + (pl.ml_tiles == 1 ? ml_bytes / 4 : ml_bytes);
    pl.ok = pl.smem_bytes <= kMaxSmem;
    pl.mode = pl.resident ? 1 : 0;
    return pl;
}

// Suffix-ring mode with tiles that end anywhere in the row list: one query head per KV head and 66 suffix keys are 66
// rows of a 128-row tile where a tile's suffix keys have to fit one block, or 120 rows and two or three suffix blocks.
TilePlan plan_straddle(const Dims &dm)
{
    TilePlan pl;
    memset(&pl, 0, sizeof(pl));
    int nc = 0;
    if (!pick_tile_rows(dm, true, false, &pl, &nc)) return pl;
    pl.mode = 3;
    pl.Spad = pl.Sp;
    pl.cpb = kBlockN / pl.Sp;
    pl.cbox = 1;
    layout_ring(dm, &pl);
    return pl;
}

// Estimated cycles of the SM with the most tiles.
double busiest(const Dims &dm, const TilePlan &pl)
{
    const long long sms = sm_count(), tiles = (long long)pl.tiles_per_group * dm.Hkv;
    return (double)((tiles + sms - 1) / sms) * pl.cost / pl.tiles_per_group;
}

// The full-suffix operator takes the tiling with the suffix in one block unless another one is clearly cheaper: tiles
// that straddle candidates, or, for groups of a few rows, whole candidates without padding (one row per candidate and
// head padded to 8 would be an eighth of the tile).  The decode-shaped operator and suffixes beyond one block are the
// suffix-ring mode's.  Straddling tiles fetch the prefix for every tile, so they have to be cheaper by 40 % by count of
// blocks where it would stay resident (B = 74, 32/8 heads, P = 256, S = 75: 57 us instead of 49 at a count 12 %
// lower), by 8 % where it is streamed either way (B = 58, 32/32, P = 1735, S = 66 221 -> 168 us; B = 66, 32/8, P = 803,
// S = 109 152 -> 145), on the whole and on the SM with the most tiles: fewer tiles gain nothing where they take as many rounds
// (B = 65, 4/4, P = 1183, S = 81 33.3 us straddling, 25.6 not; B = 35, 8/2, P = 315, S = 67 16.7 and 12.8), and a round less
// is not enough by itself (B = 23, 8/8, P = 365, S = 84 13.8 and 13.2).
TilePlan make_plan(const Dims &dm, int n_instr)
{
    if (dm.Skv == dm.S && !dm.ragged) {
        const TilePlan pl = plan_base(dm, n_instr > 1);
        if (n_instr > 1) return pl;  // (several instructions in one launch: only this tiling)
        if (pl.ok && dm.n_rep * dm.S % 8 != 0 && dm.n_rep * dm.S <= kTileM / 2) {
            const TilePlan ring = plan_suffix_ring(dm);
            if (ring.ok && !ring.long_sfx && ring.cost < pl.cost) return ring;
        }
        if (pl.ok) {
            const TilePlan ring = plan_straddle(dm);
            const double margin = pl.resident ? 1.4 : 1.08;
            return ring.ok && margin * ring.cost < pl.cost && margin * busiest(dm, ring) < busiest(dm, pl) ? ring : pl;
        }
    }
    return plan_suffix_ring(dm);
}

const TilePlan &plan_tiles(const Dims &dm, int n_instr = 1)
{
    static thread_local PlanTable<TilePlan> table;
    return table.get(dm, n_instr, [&] { return make_plan(dm, n_instr); });
}

// CTAs for tiles that are dealt out by cost.  All SMs for a launch by itself: the 512 tiles of a prompt of 2048 tokens, 32 heads, put
// 34 key blocks on the busiest of 128 CTAs of four tiles, 31 on the busiest of 148 (49.5 -> 45.5 us).  `passes` such launches on
// two streams fill each other's free SMs, and a CTA's start is paid for each: counted in tiles in a row, the even grid
// takes its CTAs in waves; on all SMs a pass takes something between its tiles per SM and the most that an SM gets.  Even and all: 4
// passes of 192 tiles (2 candidates, 32/32 heads, P = 128, S = 384) 49.0 and 56.1 us, 8 of 192 (3, 32/8, P = 100, S = 256) 83 and 96, 5 of 192
// (3, 32/8, P = 64, S = 200) 55.3 and 61.6; 3 of 320 (2, 32/8, P = 500, S = 640) 86 and 71, 4 of 512 (1, 32/8, P = 64, S = 2048) 191 and 175,
// 2 of 320 (2, 32/32, P = 300, S = 520) 51.6 and 45.1; 4 of 288 (3, 32/8, P = 64, S = 384) 59.8 both.
int dealt_grid(int tiles, int sms, int passes)
{
    const int even = even_grid(tiles, sms), in_a_row = (tiles + sms - 1) / sms;
    const double waves = (double)(((long long)passes * even + sms - 1) / sms);
    return passes * 0.5 * ((double)tiles / sms + in_a_row) < waves * in_a_row ? (tiles < sms ? tiles : sms) : even;
}

template <int D>
cudaError_t launch(const FwdArgs &a, const TilePlan &plan, void *workspace, unsigned int *status_word,
                   cudaStream_t stream, int n_instr, const int *prefix_len, int passes)
{
    const Dims &dm = a.dims;
    const int Rg = dm.n_rep * dm.S;
    CUtensorMap tm_q, tm_out, tm_pk, tm_pv, tm_pk_tail, tm_pv_tail, tm_sk, tm_sv;
    memset(&tm_pk, 0, sizeof(tm_pk));
    memset(&tm_pv, 0, sizeof(tm_pv));
    memset(&tm_pk_tail, 0, sizeof(tm_pk_tail));
    memset(&tm_pv_tail, 0, sizeof(tm_pv_tail));
    {
        // q / out viewed as [B][Hkv][Rg][D]: the n_rep heads of a KV head are contiguous rows
        cuuint64_t dims[4] = {(cuuint64_t)D, (cuuint64_t)Rg, (cuuint64_t)dm.Hkv, (cuuint64_t)dm.B};
        cuuint64_t str[3] = {(cuuint64_t)D * 2, (cuuint64_t)Rg * D * 2, (cuuint64_t)dm.Hkv * Rg * D * 2};
        cuuint32_t box[4] = {64, (cuuint32_t)plan.seg_rows, 1, 1};
        if (plan.head_box) {  // heads of their own
            dims[1] = (cuuint64_t)dm.S;
            dims[2] = (cuuint64_t)dm.Hq;
            str[1] = (cuuint64_t)dm.S * D * 2;
        } else if (plan.mode >= 2 && plan.one_box) {  // one box = the whole candidates of a tile, or the tile's rows of one candidate
            box[1] = (cuuint32_t)(plan.long_sfx ? plan.tile_rows : Rg);
            box[3] = (cuuint32_t)plan.cbox;
        }
        if (!encode_map(&tm_q, a.q, 4, dims, str, box)) return cudaErrorInvalidValue;
        if (!encode_map(&tm_out, a.out, 4, dims, str, box)) return cudaErrorInvalidValue;
    }
    {
        cuuint64_t dims[4] = {(cuuint64_t)D, (cuuint64_t)dm.Skv, (cuuint64_t)dm.Hkv, (cuuint64_t)dm.B};
        cuuint64_t str[3] = {(cuuint64_t)D * 2, (cuuint64_t)dm.Skv * D * 2, (cuuint64_t)dm.Hkv * dm.Skv * D * 2};
        cuuint32_t box[4] = {64, (cuuint32_t)(plan.long_sfx ? kBlockN : plan.mode >= 2 ? dm.Skv : plan.Sp), 1, 1};
        if (!encode_map(&tm_sk, a.suffix_k, 4, dims, str, box)) return cudaErrorInvalidValue;
        if (!encode_map(&tm_sv, a.suffix_v, 4, dims, str, box)) return cudaErrorInvalidValue;
    }
    if (dm.P > 0) {
        cuuint64_t dims[3] = {(cuuint64_t)D, (cuuint64_t)dm.P, (cuuint64_t)dm.Hkv * (cuuint64_t)n_instr};
        cuuint64_t str[2] = {(cuuint64_t)D * 2, (cuuint64_t)dm.Pstride * D * 2};
        cuuint32_t box[3] = {64, (cuuint32_t)kBlockN, 1};
        cuuint32_t box_tail[3] = {64, (cuuint32_t)plan.tail_rows, 1};
        if (!encode_map(&tm_pk, a.prefix_k, 3, dims, str, box)) return cudaErrorInvalidValue;
        if (!encode_map(&tm_pv, a.prefix_v, 3, dims, str, box)) return cudaErrorInvalidValue;
        if (!encode_map(&tm_pk_tail, a.prefix_k, 3, dims, str, box_tail)) return cudaErrorInvalidValue;
        if (!encode_map(&tm_pv_tail, a.prefix_v, 3, dims, str, box_tail)) return cudaErrorInvalidValue;
    }
    // one instantiation: its parameters and its launch
    auto run = [&](auto kernel, auto &&p, int slot) {
        p.lse = a.lse;
        p.status = status_word;
        p.args = a;
        p.sl2 = a.scale * kLog2e;
        p.B = dm.B; p.Hq = dm.Hq; p.Hkv = dm.Hkv; p.S = dm.S; p.P = dm.P; p.n_rep = dm.n_rep;
        p.Rg = plan.Rp;
        p.box.Sh = plan.head_box ? plan.Sh : dm.S;
        p.Rr = dm.n_rep * p.box.Sh;
        p.box.one_box = plan.one_box;
        p.box.head_box = plan.head_box;
        p.Sp = plan.mode >= 2 ? dm.S : plan.Sp;
        p.tile_rows = plan.tile_rows;
        p.seg_rows = plan.seg_rows;
        p.fd_Rg.init(p.Rg);
        p.fd_S.init(p.box.Sh);
        p.fd_seg.init(plan.seg_rows);
        p.nblk_p = plan.nblk_p;
        p.tail_rows = plan.tail_rows;
        p.resident = plan.resident;
        p.stages = plan.stages > 0 ? plan.stages : 1;
        p.sfx_rows = plan.sfx_rows;
        p.alias_stage = plan.alias_stage;
        p.slab_stage = plan.slab_stage;
        p.ml_mask = plan.ml_tiles == 1 ? 0 : 3;
        p.suffix_len = a.suffix_len;
        p.Skv = dm.Skv;
        p.Spad = plan.Spad > 0 ? plan.Spad : 8;
        p.cpb = plan.cpb > 0 ? plan.cpb : 1;
        p.fd_cpb.init(p.cpb);
        p.long_sfx = plan.long_sfx;
        p.n_instr = n_instr;
        p.rpi = dm.B / n_instr * p.Rg;
        p.fd_rpi.init(p.rpi > 0 ? p.rpi : 1);
        p.tpi = n_instr > 1 ? (p.rpi + plan.tile_rows - 1) / plan.tile_rows : plan.tiles_per_group;
        p.fd_tpi.init(p.tpi);
        p.tiles_per_group = p.tpi * n_instr;
        p.fd_tpg.init(p.tiles_per_group);
        p.total_tiles = p.tiles_per_group * dm.Hkv;
        for (int i = 0; i < kMaxInstr; ++i) p.pad[i] = (n_instr > 1 && i < n_instr) ? dm.P - prefix_len[i] : 0;
        // Dealing by cost balances the causal skew but lets every CTA touch every candidate's suffix K/V
        // at several times; it pays when those tensors stay in L2 between the touches.
        p.deal_by_cost = plan.long_sfx && p.box.Sh % plan.tile_rows == 0 && p.box.Sh / plan.tile_rows > 1 &&
                         4.0 * dm.B * dm.Hkv * dm.Skv * D <= 48.0e6;
        p.off_pk = plan.off_pk; p.off_pv = plan.off_pv; p.off_q = plan.off_q; p.off_sk = plan.off_sk;
        p.off_sv = plan.off_sv; p.off_stage = plan.off_stage; p.off_bar = plan.off_bar; p.off_misc = plan.off_misc;
        p.off_ml = plan.off_ml;
        // The MMAs read keys in steps of 16: candidates that take a multiple of 16 leave no row of a block unwritten, and
        // the boxes of prefix and long-suffix blocks are whole blocks, filled with zeros past the end.
        p.zero_lo = p.zero_hi = 0;
        if (plan.mode >= 2) {
            if (!plan.long_sfx && dm.Skv % 16 != 0) p.zero_lo = plan.off_pv, p.zero_hi = plan.off_q;
        } else if (plan.Sp % 16 != 0) {
            p.zero_lo = plan.off_sv, p.zero_hi = plan.off_sv + D / 64 * plan.sfx_rows * 128;
        }

        static PerDeviceOnce attr_set[9];
        if (cudaError_t e = ensure_max_smem(kernel, attr_set[slot]); e != cudaSuccess) return e;
        const int grid = p.deal_by_cost ? dealt_grid(p.total_tiles, sm_count(), passes) : even_grid(p.total_tiles, sm_count());
        cudaError_t launch_err;
        {
            KernelTiming timing(kKernelFwdTc, stream);
            launch_err = launch_dependent(kernel, grid, kThreads, plan.smem_bytes, stream, tm_q, tm_out, tm_pk, tm_pv, tm_pk_tail,
                                          tm_pv_tail, tm_sk, tm_sv, p);
        }
        count_launches(1);
        return launch_err != cudaSuccess ? launch_err : cudaGetLastError();
    };
    if (n_instr > 1) {  // (never with the suffix-ring tiling) whole tiles of every instruction, or the last one of each short
        const bool whole = (long long)(dm.B / n_instr) * plan.Rp % plan.tile_rows == 0;
        if (whole) return plan.mode == 1 ? run(tc_fwd_kernel<D, 1, 1>, TcFwdParams<1>(), 4) : run(tc_fwd_kernel<D, 0, 1>, TcFwdParams<1>(), 5);
        return plan.mode == 1 ? run(tc_fwd_kernel<D, 1, 2>, TcFwdParams<2>(), 6) : run(tc_fwd_kernel<D, 0, 2>, TcFwdParams<2>(), 7);
    }
    if (plan.mode == 3 && plan.two_terms) return run(tc_fwd_kernel<D, 3, 0, true>, TcFwdParams<0>(), 8);
    return run(plan.mode == 3 ? tc_fwd_kernel<D, 3, 0> : plan.mode == 2 ? tc_fwd_kernel<D, 2, 0> : plan.mode == 1 ? tc_fwd_kernel<D, 1, 0>
                                                                                                             : tc_fwd_kernel<D, 0, 0>,
               TcFwdParams<0>(), plan.mode);
}

}  // namespace

#ifdef PSKV_TRACE
// Debug builds only: copies the event trace of CTA 0 to the host (all warps' events concatenated).
extern "C" int pskv_debug_read_trace(long long *host, int max_events)
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

bool tc_fwd_supported(const Dims &dm)
{
    if (dm.d != 64 && dm.d != 128) return false;
    if ((long long)dm.B * dm.n_rep * dm.S > 2000000000ll) return false;  // flat row index fits an int
    const TilePlan &pl = plan_tiles(dm);
    return pl.ok && (long long)pl.tiles_per_group * dm.Hkv <= 2000000000ll;  // ... and so does the tile index
}

size_t tc_fwd_workspace_bytes(const Dims &) { return 0; }

// One launch can serve several instructions when the tiles are those with one suffix block each (not the suffix-ring
// tiling).  An instruction starts a tile of its own, so its last tile may be short: taken where an instruction is a
// whole number of tiles, or at least four, so that the short one costs at most a fifth (90 candidates of 6
// instructions, 32/8 heads, P = 300, S = 37: one launch 107 us for forward + backward, six passes
// on two streams 131, the gradients in one term both times).
bool tc_fwd_fused_supported(const Dims &dm, int n_instr)
{
    if (n_instr < 2 || n_instr > kMaxFusedInstructions || dm.B % n_instr != 0 || dm.P < 1 || dm.Pstride != dm.P ||
        dm.ragged || !tc_fwd_supported(dm))
        return false;
    const TilePlan &pl = plan_tiles(dm, n_instr);
    const long long rows = (long long)(dm.B / n_instr) * pl.Rp;
    return pl.ok && pl.mode < 2 && (rows % pl.tile_rows == 0 || rows >= 4 * pl.tile_rows) &&
           (rows / pl.tile_rows + 1) * n_instr * dm.Hkv <= 2000000000ll;
}

cudaError_t launch_tc_fwd(const FwdArgs &a, void *workspace, unsigned int *status_word, cudaStream_t stream,
                          int n_instr, const int *prefix_len, int passes)
{
    if (n_instr < 1) n_instr = 1;
    const TilePlan plan = plan_tiles(a.dims, n_instr);  // (a copy: the next look-up may replace the table's entry)
    if (!plan.ok) return cudaErrorInvalidValue;
    if (n_instr > 1 && (!prefix_len || !tc_fwd_fused_supported(a.dims, n_instr))) return cudaErrorInvalidValue;
    if (n_instr == 1 && cta_pairs_enabled() && tc_fwd_pair_supported(a.dims))
        return launch_tc_fwd_pair(a, status_word, stream);
    return a.dims.d == 128 ? launch<128>(a, plan, workspace, status_word, stream, n_instr, prefix_len, passes)
                           : launch<64>(a, plan, workspace, status_word, stream, n_instr, prefix_len, passes);
}

}  // namespace pskv
