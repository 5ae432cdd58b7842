// Wide-block variant of the tensor-core GEMM  Y[m, N] = X[m, K] . W[N, K]^T  for up to
// CSD_WIDE_ROWS rows: the prompt prefill and the encoder pass, where the model takes many tokens in
// one run (Section 2) and the weights should stream once per pass.
//
// Each fp32 value of X enters as TWO bf16 terms x = hi + lo (16 mantissa bits, relative error
// 2^-17), laid out as [2][mpad][K].  A tile is 256 weight rows x nt <= 256 tokens (the gated pair:
// 128 rows of each matrix, or up to 64 tokens 256 rows of each) and belongs to a PAIR of CTAs on
// neighbouring SMs: tcgen05.mma with cta_group::2, 128 weight rows and half of the tokens' terms staged by
// each CTA; both terms are accumulated into the same fp32 columns, up to 128 tokens side by side.
//
// What bounds it: beyond 128 tokens the MMAs and what they read from shared memory (a full tile: 112 KB per 1024 tensor clocks and SM, of
// 128 KB that it can give; copies into it 48 KB, where each of 148 SMs can draw 130 GB/s from L2), under the power limit;
// 1024 rows, N 12288, K 4096: MMAs alone 89 us, the kernel 157 us (1.29 PFLOP/s of two-term products, 77 % of the measured one-term cuBLAS
// rate).  Up to 128 tokens the weight stream and, since a CTA fills an SM, each launch's start from an empty ring and its finish:
// q|k|v of the 7B shape at 64 tokens 28 us, of which 18 are the stream.
//
// fp32 accumulation.  The tensor core loses a little with every add of a long chain, so after WG_DRAIN
// K blocks (64 adds) the accumulator set is added into fp32 registers of the epilogue warps while
// the MMAs continue on the other set, and the epilogue of one tile overlaps the MMAs of the next.  Error against fp64 at K = 4096 to
// 12288 (csd_linear, 18 to 128 rows, where the low terms' products have columns of their own): 2.50e-6, of which the two-term form
// itself leaves 2.45e-6; both terms in one chain 2.7e-6.  Sets of 4 K blocks, which leave 2.5e-6 either way, cost 2 to 7 % a GEMM.
//
// Roles inside a CTA (384 threads): lane 0 of warp 0 issues TMA (up to 128 tokens and for parts of K lane 0 of warp 2 that of the row
// terms), warp 1 lane 0 of the pair's first CTA issues the MMAs for both, warps 4-11 read tensor memory (two warps per quadrant, each half of the
// tokens) and finish tiles; they hold 128 accumulators each, hence the register split.  Every
// mbarrier wait is bounded; on a time-out the CTA records CSD_ERR_TIMEOUT, stops, frees its tensor
// memory, returns.
#include "gemm_tc.cuh"
#include "tc_common.cuh"

namespace csd {

constexpr size_t WG_SMEM_MAX = 227 * 1024;
constexpr int WG_MAX_STAGES = 10;
constexpr int WG_THREADS = 384;              // one control warpgroup, two epilogue warpgroups
// Registers a thread: 168 at launch (65536 / 384); 128 x 72 + 256 x 216 = 384 x 168.  Without the split the
// accumulators spill.
constexpr int WG_REGS_CTL = 72, WG_REGS_EPI = 216;
constexpr int WG_ROWS = 256;                 // weight rows of a pair's tile
constexpr int WG_DRAIN = 8;                  // K blocks per accumulator set before it is added into registers
constexpr int WG_MAX_PARTS = 8;              // most parts of K a tile goes by
constexpr int WG_SET = 256;                  // tensor-memory columns of a set

struct __align__(8) WgCtrl {
    uint64_t full[WG_MAX_STAGES], empty[WG_MAX_STAGES], acc_full[2], acc_empty[2];
    uint64_t part_full;                      // parked partial sums have landed in the ring
    uint32_t tmem_base;
    int abort_flag;
    float scale[256];                        // rms-norm factors of the tile's tokens
};
// Epilogue staging: a warp's 32 weight rows x 16 tokens (of both matrices of a gated pair).  An accumulator thread owns one
// weight row, memory wants the rows of a token side by side.  A single matrix's second half holds the pieces of the
// sums of squares (one float per quadrant and token).
constexpr size_t WG_STAGING = 2 * 8 * 16 * 32 * sizeof(float);
static_assert(8 * 16 * 32 + 4 * WG_SET <= 2 * 8 * 16 * 32, "sums of squares fit behind the staging of a single matrix");

// How a launch is divided.  tiles = row tiles x token tiles, tokens fastest, so that pairs running at the
// same time share weight rows in L2.  Three ways:
//   parts    few tiles of a single matrix (at most half as many as pairs): every tile goes to pk pairs that share its K range.
//            Each of them finishes a pk-th of the tile's tokens and parks its sums of the others' (they stay in L2).  With fp32
//            planes and a kernel behind that added them and ran the epilogue, the GEMM after o and down of a 7B-shaped
//            layer of 64 tokens met its rows 9.7 us after their end.  A layer of 64 / 128 / 256 tokens 133 -> 129, 160 -> 145,
//            245 -> 235 us; two parts instead of shares: 512 tokens 454 -> 440, eight T5-xxl-shaped encoder layers of 128 1326 -> 1291.
//            (Clusters of four pairs that add up through distributed shared memory: 15 of them are resident, for 16 tiles.)
//            A tile's pairs wait for one another, so all of them must come to be resident: they are neighbours in a grid that is dispatched
//            in order, so of a launch that shares the GPU at most one tile waits for places, which the tiles before it give back;
//   whole    pair c takes whole tiles (no partial sums) where that leaves little of the last round empty;
//   shares   otherwise the (tile, K block) units are dealt out in equal contiguous shares; a tile cut by a
//            share boundary is finished by its first contributor from the partial sums the later
//            ones parked before they went on (the same scheme, and the same order of waiting, as in
//            gemm_tc.cu).
// whole or shares: by the K blocks of the busiest pair, a fix-up (park, fetch, add: about 5 us) counted as 8 blocks
// of a full tile (0.55 us each).
struct WgPlan {
    int mpad, nt, ntok, tiles, nkb, pairs, pk, gran, stages;
    bool merged;                             // both terms of a tile's tokens in one MMA (up to 128 tokens)
    bool mixed;                              // gated pair: a tile's weight rows are half gate, half up
    size_t stage, smem;
};

int wide_split_pieces(int K) { return (K + 1023) / 1024; }

static WgPlan wg_plan(int m, int N, int K, bool dual) {
    WgPlan p{};
    const int P = tc_sm_count() / 2, most = 256;
    p.mixed = dual && m > 64;
    const int rows = p.mixed ? WG_ROWS / 2 : WG_ROWS;
    p.mpad = (m + 15) & ~15;
    p.ntok = (m + most - 1) / most;
    p.nt = ((m + p.ntok - 1) / p.ntok + 31) & ~31;
    p.merged = p.nt <= 128;
    p.tiles = ((N + rows - 1) / rows) * p.ntok;
    p.nkb = (K + KB - 1) / KB;
    p.stage = (size_t)STAGE_BYTES * (dual && !p.mixed ? 2 : 1) + (size_t)p.nt * 128;
    p.stages = (int)((WG_SMEM_MAX - 1024 - WG_STAGING - sizeof(WgCtrl)) / p.stage);
    if (p.stages > WG_MAX_STAGES) p.stages = WG_MAX_STAGES;
    p.smem = (size_t)p.stages * p.stage + 1024 + WG_STAGING + sizeof(WgCtrl);
    p.pk = 1; p.gran = 1;
    const int ratio = P / p.tiles;
    if (!dual && ratio >= 2 && p.nkb >= 16) {
        p.pk = ratio < WG_MAX_PARTS ? ratio : WG_MAX_PARTS;
        if (p.pk > p.nkb / 8) p.pk = p.nkb / 8;
        p.pairs = p.tiles * p.pk;
        return p;
    }
    const double kb = (double)p.nkb, fix = 8.0;
    const double whole = (double)((p.tiles + P - 1) / P) * kb, shares = (double)p.tiles * kb / P + fix;
    if (whole <= shares) {
        p.gran = p.nkb;
        p.pairs = p.tiles < P ? p.tiles : P;
    } else {
        const long long units = (long long)p.tiles * p.nkb;
        p.pairs = units / 4 < P ? (int)(units / 4 > 0 ? units / 4 : 1) : P;
    }
    return p;
}

bool wide_supported(int m, int N, int K, bool dual) {
    (void)dual;
    if (m < 1 || m > CSD_WIDE_ROWS || N < 1 || K < 64 || (K & 7)) return false;
    if ((long long)N * K < (1LL << 20)) return false;
    const long long tiles = (long long)((N + WG_ROWS / 2 - 1) / (WG_ROWS / 2)) * ((m + 127) / 128);
    return tiles * ((K + KB - 1) / KB) * (tc_sm_count() + 1) < (1LL << 31);
}

int wide_ssq_pieces(int N) { return 2 * ((N + WG_ROWS - 1) / WG_ROWS); }
// one parked tile (of both matrices of a gated pair) per pair
size_t wide_partial_bytes(int m) {
    const int cols = m < 128 ? 2 * ((m + 31) & ~31) : 256;
    return (size_t)(tc_sm_count() / 2) * WG_ROWS * cols * sizeof(float);
}
int wide_ticket_count(int m, int N) {
    const int half = WG_ROWS / 2;
    const int a = ((N + WG_ROWS - 1) / WG_ROWS) * ((m + 127) / 128), b = ((N + half - 1) / half) * ((m + 255) / 256);
    const int tiles = a > b ? a : b, pairs = tc_sm_count() / 2;
    const int parts = WG_MAX_PARTS * tiles < pairs ? WG_MAX_PARTS * tiles : pairs;      // most pairs where tiles go by parts
    return 2 * (tiles > parts ? tiles : parts);                                         // two words a tile, or a pair
}

struct WgParams {
    float* Y; float* partial; unsigned* tickets; int* status;
    const float* ssq_in; int ssq_cnt;
    __nv_bfloat16* out_xs; const __nv_bfloat16* out_gain; float* out_ssq; int out_ld;
    int m, mpad, nt, ntok, tiles, nkb, pk, gran, N, K, ldy, stages, epilogue;
    int vec_y;                          // Y takes 16-byte accesses
    float eps;
};

// x = hi + lo with bf16 terms (16 mantissa bits)
__device__ __forceinline__ void split2f(float x, uint16_t& hi, uint16_t& lo) {
    hi = float_to_bf16_bits(x);
    lo = float_to_bf16_bits(x - bf16_bits_to_float(hi));
}

// ---- the pair's forms of the tensor-core instructions ---------------------------------------------
// a copy into this CTA's shared memory that completes on the barrier at cluster address `bar`
__device__ __forceinline__ void tma_load_2d_pair(void* dst, const CUtensorMap* tm, uint32_t bar, int x, int y) {
    asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes.cta_group::2 [%0], [%1, {%3, %4}], [%2];"
                 ::"r"(smem_u32(dst)), "l"((uint64_t)tm), "r"(bar), "r"(x), "r"(y) : "memory");
}
__device__ __forceinline__ void tma_load_2d_pair_hint(void* dst, const CUtensorMap* tm, uint32_t bar, int x, int y, uint64_t pol) {
    asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes.cta_group::2.L2::cache_hint [%0], [%1, {%3, %4}], [%2], %5;"
                 ::"r"(smem_u32(dst)), "l"((uint64_t)tm), "r"(bar), "r"(x), "r"(y), "l"(pol) : "memory");
}
__device__ __forceinline__ void tc_mma_pair(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t accum) {
    asm volatile("{ .reg .pred p; setp.ne.b32 p, %4, 0; tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p; }"
                 ::"r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accum) : "memory");
}
// arrives at the barrier of this offset in both CTAs once the MMAs issued before have finished
__device__ __forceinline__ void tc_commit_pair(uint64_t* bar) {
    asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
                 ::"r"(smem_u32(bar)), "h"((uint16_t)3) : "memory");
}
// 1D copy from global into this CTA's shared memory (16-byte aligned on both sides, a multiple of 16 bytes)
__device__ __forceinline__ void bulk_to_smem(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(smem_u32(dst)), "l"(src), "r"(bytes), "r"(smem_u32(bar)) : "memory");
}

// first unit of pair c: equal shares of `gran` units each
__device__ __forceinline__ unsigned wg_begin(unsigned c, unsigned units, unsigned pairs, unsigned gran) {
    return unit_begin(c, units / gran, pairs) * gran;
}

// MODE 0: one matrix; 1: a gated pair, both matrices' 256 rows in a stage (up to 64 tokens); 2: a gated pair, the CTA's
// 128 rows are 64 of the gate and the same 64 of the up matrix, so that the MMAs are up to 256 columns wide.  (An MMA reads
// its 128 weight rows from shared memory whatever its width, and those reads, not the tensor pipe, set the pace of narrow ones.)
// MERGED (tiles of up to 128 tokens): one MMA multiplies both terms of the tile's tokens, 2 nt columns wide, the high terms'
// sums in the first nt columns and the low terms' in the others; one CTA of the pair stages the high terms of all tokens, the
// other the low ones.  An MMA of 256 x 64 takes little less time than one of 256 x 128, so two of them per term and K step set
// the pace of small tiles (0.46 to 0.49 us a K block of a single matrix, whatever the tokens; weights alone need 0.37).  A layer
// of the 7B shape at 20 / 64 / 128 tokens 134 -> 120, 151 -> 133, 173 -> 160 us; eight layers of the T5-xxl-shaped encoder at 64 /
// 128 tokens 1373 -> 1217, 1568 -> 1385 us.  The gated pair at 100 / 128 tokens of that in mode 1, terms apart: 155 (7B), 1427 (T5);
// in mode 2, merged: 150, 1385.
template <int MODE, bool MERGED, bool PARTS>
__global__ void __launch_bounds__(WG_THREADS, 1)
wide_gemm_kernel(const __grid_constant__ CUtensorMap tmW, const __grid_constant__ CUtensorMap tmW2,
                 const __grid_constant__ CUtensorMap tmX, const WgParams p) {
    constexpr bool DUAL = MODE == 1, MIXED = MODE == 2;
    constexpr int NT = DUAL ? 2 : 1;
    constexpr int OUT_ROWS = MIXED ? WG_ROWS / 2 : WG_ROWS;   // outputs of a tile
    constexpr uint32_t WB = NT * STAGE_BYTES;                 // weight bytes per stage and CTA
    static_assert(MODE != 1 || MERGED, "both matrices' sums of both terms fit a set up to 64 tokens");
    constexpr int CH = MERGED ? (DUAL ? 2 : 4) : 8;           // 16-token chunks an epilogue warp holds at most
    const int nt = p.nt, htok = nt >> 1;
    const uint32_t mma_cols = MERGED ? 2 * nt : nt;           // columns of an MMA
    const uint32_t xterm = (uint32_t)htok * 128u;             // one term of this CTA's half of the tokens
    const uint32_t stage_bytes = WB + 2u * xterm;
    const uint32_t IDESC = (1u << 4) | (1u << 7) | (1u << 10) | ((mma_cols >> 3) << 17) |
                           ((uint32_t)(WG_ROWS >> 4) << 24);  // f32 accumulate, bf16 x bf16, K-major both

    extern __shared__ unsigned char smem_raw[];
    unsigned char* ring = (unsigned char*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    float* staging = (float*)(ring + (size_t)p.stages * stage_bytes);
    WgCtrl* ctl = (WgCtrl*)((unsigned char*)staging + WG_STAGING);

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int rank = (int)(blockIdx.x & 1), pair = (int)(blockIdx.x >> 1), pairs = (int)(gridDim.x >> 1);
    const unsigned units = (unsigned)p.tiles * (unsigned)p.nkb;
    unsigned u0, u1;
    if (PARTS) {
        const unsigned t = (unsigned)(pair / p.pk) * (unsigned)p.nkb, part = (unsigned)(pair % p.pk);
        u0 = t + part * (unsigned)p.nkb / (unsigned)p.pk;
        u1 = t + (part + 1) * (unsigned)p.nkb / (unsigned)p.pk;
    } else {
        u0 = wg_begin(pair, units, pairs, p.gran);
        u1 = wg_begin(pair + 1, units, pairs, p.gran);
    }
    const int items = (int)(u1 - u0);

    if (tid == 0) {
#pragma unroll 1
        for (int s = 0; s < WG_MAX_STAGES; ++s) { mbar_init(&ctl->full[s], 1); mbar_init(&ctl->empty[s], 1); }
        for (int b = 0; b < 2; ++b) { mbar_init(&ctl->acc_full[b], 1); mbar_init(&ctl->acc_empty[b], 16); }
        mbar_init(&ctl->part_full, 1);
        ctl->abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(smem_u32(&ctl->tmem_base)), "r"((uint32_t)(2 * WG_SET)) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    cluster_barrier();               // nobody signals a barrier of the other CTA before it is initialised
    tc_fence_after();
    const uint32_t tmem = ctl->tmem_base;
    volatile int* abort_flag = &ctl->abort_flag;
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

    if (warp < 4) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(WG_REGS_CTL));
        struct Cursor { int kb, row, tok; };                  // K block, row tile, token tile
        auto step = [&](Cursor& c) {
            if (++c.kb == p.nkb) { c.kb = 0; if (++c.tok == p.ntok) { c.tok = 0; ++c.row; } }
        };
        auto first = [&] {
            const int tile0 = (int)(u0 / p.nkb);
            return Cursor{(int)(u0 % p.nkb), tile0 / p.ntok, tile0 % p.ntok};
        };
        // All copies of the pair complete on the first CTA's barriers.
        auto load_w = [&](int s, const Cursor& c, uint64_t once) {
            unsigned char* dst = ring + (size_t)s * stage_bytes;
            const uint32_t bar = map_to_cta(smem_u32(&ctl->full[s]), 0u);
            if (rank == 0) mbar_expect_tx(&ctl->full[s], 2u * stage_bytes);
            const int row = c.row * OUT_ROWS + rank * (OUT_ROWS / 2);
            if (p.ntok == 1) {                                // no other token tile takes these weights from L2
                tma_load_2d_pair_hint(dst, &tmW, bar, c.kb * KB, row, once);
                if (DUAL) tma_load_2d_pair_hint(dst + STAGE_BYTES, &tmW2, bar, c.kb * KB, row, once);
                if (MIXED) tma_load_2d_pair_hint(dst + STAGE_BYTES / 2, &tmW2, bar, c.kb * KB, row, once);
            } else {
                tma_load_2d_pair(dst, &tmW, bar, c.kb * KB, row);
                if (DUAL) tma_load_2d_pair(dst + STAGE_BYTES, &tmW2, bar, c.kb * KB, row);
                if (MIXED) tma_load_2d_pair(dst + STAGE_BYTES / 2, &tmW2, bar, c.kb * KB, row);
            }
        };
        auto load_x = [&](int s, const Cursor& c) {           // this CTA's half of the row terms
            unsigned char* dst = ring + (size_t)s * stage_bytes + WB;
            const uint32_t bar = map_to_cta(smem_u32(&ctl->full[s]), 0u);
            if (MERGED) {
                tma_load_2d_pair(dst, &tmX, bar, c.kb * KB, rank * p.mpad + c.tok * nt);
            } else {
                const int r = c.tok * nt + rank * htok;
                tma_load_2d_pair(dst, &tmX, bar, c.kb * KB, r);
                tma_load_2d_pair(dst + xterm, &tmX, bar, c.kb * KB, p.mpad + r);
            }
        };
        // The row terms come from a warp of their own where a K block is short: three copies a stage from one thread (about 100 ns each,
        // with the wait before them) set the pace of tiles of up to 128 tokens.  Full tiles whose weights several token tiles share gain
        // nothing, and under the power limit a second thread and a cache hint cost: prompts of the 7B shape at 513 / 700 / 768 tokens
        // +0.8 / +0.9 / +0.9 %, one thread +0.65 / +0.4 / +0.4, and no hint level.
        constexpr bool TWO = MERGED || PARTS;
        if (warp == 0 && lane == 0) {
            // ---- TMA producer of this CTA's weights, or of all it stages
            const uint64_t once = policy_evict_first();
            Cursor cw = first(), cx = cw;
            const int pre = items < p.stages ? items : p.stages;
#pragma unroll 1
            for (int i = 0; i < pre; ++i) { load_w(i, cw, once); step(cw); }
            if (!TWO) {
                asm volatile("griddepcontrol.wait;" ::: "memory");
#pragma unroll 1
                for (int i = 0; i < pre; ++i) { load_x(i, cx); step(cx); }
            }
            int s = 0;
            uint32_t ph = 0;
#pragma unroll 1
            for (int i = pre; i < items && !*abort_flag; ++i) {
                if (!mbar_wait(&ctl->empty[s], ph)) { *abort_flag = 1; break; }
                load_w(s, cw, once);
                step(cw);
                if (!TWO) { load_x(s, cx); step(cx); }
                if (++s == p.stages) { s = 0; ph ^= 1u; }
            }
        } else if (TWO && warp == 2 && lane == 0) {
            // ---- TMA producer of its row terms
            asm volatile("griddepcontrol.wait;" ::: "memory");
            Cursor cx = first();
            int s = 0;
            uint32_t ph = 0;
#pragma unroll 1
            for (int i = 0; i < items && !*abort_flag; ++i) {
                if (i >= p.stages && !mbar_wait(&ctl->empty[s], ph)) { *abort_flag = 1; break; }
                load_x(s, cx);
                step(cx);
                if (++s == p.stages) { s = 0; if (i >= p.stages) ph ^= 1u; }
            }
        } else if (warp == 1 && rank == 0 && lane == 0) {
            // ---- MMA issuer of the pair
            int s = 0, i = 0;
            uint32_t ph = 0;
            int kb_begin = (int)(u0 % p.nkb);
            unsigned g = 0;                                   // accumulator sets filled so far
            const uint64_t desc0 = smem_desc_sw128(smem_u32(ring));
#pragma unroll 1
            while (i < items && !*abort_flag) {
                int left = min(p.nkb - kb_begin, items - i);  // K blocks of this segment
                kb_begin = 0;
#pragma unroll 1
                while (left > 0) {
                    const int b = g & 1, cnt = min(left, WG_DRAIN);
                    if (!mbar_wait(&ctl->acc_empty[b], ((g >> 1) & 1) ^ 1)) { *abort_flag = 1; break; }
                    tc_fence_after();
                    const uint32_t d0 = tmem + (uint32_t)(b * WG_SET);
#pragma unroll 1
                    for (int j = 0; j < cnt; ++j, ++i) {
                        if (!mbar_wait(&ctl->full[s], ph)) { *abort_flag = 1; break; }
                        tc_fence_after();
                        const uint64_t ad = desc0 + (uint64_t)(((uint32_t)s * stage_bytes) >> 4);
                        const uint64_t bh = ad + (WB >> 4), bl = bh + (xterm >> 4);
#pragma unroll
                        for (int k = 0; k < KB / 16; ++k) {
                            const uint32_t acc = (j | k) != 0;
                            tc_mma_pair(d0, ad + 2 * k, bh + 2 * k, IDESC, acc);
                            if (!MERGED) tc_mma_pair(d0, ad + 2 * k, bl + 2 * k, IDESC, 1u);
                            if (DUAL) {
                                tc_mma_pair(d0 + mma_cols, ad + (STAGE_BYTES >> 4) + 2 * k, bh + 2 * k, IDESC, acc);
                                if (!MERGED) tc_mma_pair(d0 + mma_cols, ad + (STAGE_BYTES >> 4) + 2 * k, bl + 2 * k, IDESC, 1u);
                            }
                        }
                        tc_commit_pair(&ctl->empty[s]);
                        if (++s == p.stages) { s = 0; ph ^= 1u; }
                    }
                    if (*abort_flag) break;
                    tc_commit_pair(&ctl->acc_full[b]);
                    left -= cnt;
                    ++g;
                }
            }
        }
    } else {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(WG_REGS_EPI));
        // ---- epilogue warps: quadrant q of tensor memory holds weight rows q*32 .. q*32+31 of this CTA's 128;
        //      warp half `half` takes tokens half*htok .. of the tile, 16 at a time
        const int q = warp & 3, ew = warp - 4, half = ew >> 2, et = tid - 128, m = p.m;
        const int nch = nt >> 5;                              // 16-token chunks of this warp
        const uint32_t part_bytes = (uint32_t)(TILE_N * NT * sizeof(float)) * (uint32_t)nt;
        asm volatile("griddepcontrol.wait;" ::: "memory");
        const uint32_t empty_bar = map_to_cta(smem_u32(&ctl->acc_empty[0]), 0u);
        // Accumulator sets read so far; negative once this warp has waited in vain.  It then goes on through every barrier (and stores
        // what it has, under CSD_ERR_TIMEOUT): another warp's wait may still have ended well, and would wait for it there.
        int g = 0;
#pragma unroll 1
        for (int i = 0; i < items;) {
            const int tile = (int)((u0 + i) / p.nkb), kb_begin = (int)((u0 + i) % p.nkb);
            const int seg = min(p.nkb - kb_begin, items - i);
            i += seg;
            const int row_tile = tile / p.ntok, tok0 = (tile % p.ntok) * nt;
            // a tile in parts of K: this part finishes the 16-token chunks own0 .. own1 - 1
            constexpr bool cut = PARTS;
            const int chunks = nt >> 4, kpart = cut ? pair % p.pk : 0;
            const int own0 = cut ? kpart * chunks / p.pk : 0, own1 = cut ? (kpart + 1) * chunks / p.pk : 0;
            asm volatile("bar.sync 1, 256;" ::: "memory");    // everyone is past the previous tile's scale factors
            if (p.ssq_in && et < nt && tok0 + et < m) {
                float sq = 0.f;
                const float* src = p.ssq_in + tok0 + et;
#pragma unroll 8
                for (int c = 0; c < p.ssq_cnt; ++c) sq += __ldcg(src + (size_t)c * m);
                ctl->scale[et] = 1.f / sqrtf(sq / (float)p.K + p.eps);
            }
            float acc[NT * CH * 16];
#pragma unroll
            for (int e = 0; e < NT * CH * 16; ++e) acc[e] = 0.f;
#pragma unroll 1
            for (int left = seg; left > 0 && g >= 0; left -= WG_DRAIN, ++g) {
                const int b = g & 1;
                if (!mbar_wait(&ctl->acc_full[b], (uint32_t)(g >> 1) & 1u)) { *abort_flag = 1; g = -1; break; }
                tc_fence_after();
                const uint32_t taddr = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(b * WG_SET + half * htok);
#pragma unroll
                for (int u = 0; u < NT; ++u)
#pragma unroll
                    for (int ch = 0; ch < CH; ++ch)
                        if (ch < nch) {
                            float v[16];
                            tc_ld16(taddr + u * mma_cols + (uint32_t)(ch * 16), v);
#pragma unroll
                            for (int e = 0; e < 16; ++e) acc[(u * CH + ch) * 16 + e] += v[e];
                            if (MERGED) {
                                tc_ld16(taddr + u * mma_cols + (uint32_t)(nt + ch * 16), v);
#pragma unroll
                                for (int e = 0; e < 16; ++e) acc[(u * CH + ch) * 16 + e] += v[e];
                            }
                        }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) {
                    if (rank == 0) mbar_arrive(&ctl->acc_empty[b]);
                    else remote_arrive(empty_bar + (uint32_t)(b * sizeof(uint64_t)));
                }
            }
            if (!PARTS && seg < p.nkb) {
                // part of a tile: later contributors park and go on, the first one adds the parts in pair order.
                // Parked layout [warp][chunk][quarter of 16][lane][4]: 512 contiguous bytes per warp access.
                const int c_lo = cta_of_unit((unsigned)tile * p.nkb, units, pairs);
                const int c_hi = cta_of_unit((unsigned)(tile + 1) * p.nkb - 1, units, pairs);
                const uint32_t at = (uint32_t)(ew * nch * NT * 512 + lane * 4);
                if (pair != c_lo) {
                    float* dst = p.partial + (size_t)blockIdx.x * TILE_N * nt * NT + at;
#pragma unroll
                    for (int u = 0; u < NT; ++u)
#pragma unroll
                        for (int ch = 0; ch < CH; ++ch)
                            if (ch < nch) {
#pragma unroll
                                for (int e = 0; e < 4; ++e) {
                                    const float* a = acc + (u * CH + ch) * 16 + 4 * e;
                                    __stcg(reinterpret_cast<float4*>(dst + (u * nch + ch) * 512 + e * 128), make_float4(a[0], a[1], a[2], a[3]));
                                }
                            }
                    __threadfence();
                    asm volatile("bar.sync 1, 256;" ::: "memory");
                    if (et == 0) atomicAdd(&p.tickets[2 * tile + rank], 1u);
                    continue;
                }
                // The first contributor's part is the last thing of its share: all MMAs are done, the ring is free,
                // and a parked part (at most 128 KB) comes into it by one bulk copy (through registers, few
                // loads in flight beside the accumulators, it took 8 us).
                if (et == 0) {
                    const unsigned want = (unsigned)(c_hi - c_lo);
                    int spins = 0;
#pragma unroll 1
                    while (ld_acquire_gpu(&p.tickets[2 * tile + rank]) < want)
                        if (++spins > SPIN_LIMIT || *abort_flag) { *abort_flag = 1; break; }
                    p.tickets[2 * tile + rank] = 0u;          // ready for the next launch, if everyone has arrived (clear_words)
                    __threadfence();
                    asm volatile("fence.proxy.async;" ::: "memory");
                }
                const float* mine = reinterpret_cast<const float*>(ring) + at;
#pragma unroll 1
                for (int from = c_lo + 1; from <= c_hi; ++from) {
                    if (et == 0) {
                        mbar_expect_tx(&ctl->part_full, part_bytes);
                        bulk_to_smem(ring, p.partial + (size_t)(2 * from + rank) * TILE_N * nt * NT, part_bytes, &ctl->part_full);
                    }
                    if (!mbar_wait(&ctl->part_full, (uint32_t)(from - c_lo - 1) & 1u)) *abort_flag = 1;
#pragma unroll
                    for (int u = 0; u < NT; ++u)
#pragma unroll
                        for (int ch = 0; ch < CH; ++ch)
                            if (ch < nch) {
#pragma unroll
                                for (int e = 0; e < 4; ++e) {
                                    const float4 v = *reinterpret_cast<const float4*>(mine + (u * nch + ch) * 512 + e * 128);
                                    float* a = acc + (u * CH + ch) * 16 + 4 * e;
                                    a[0] += v.x; a[1] += v.y; a[2] += v.z; a[3] += v.w;
                                }
                            }
                    asm volatile("bar.sync 1, 256;" ::: "memory");    // the ring may be overwritten
                }
            } else if (PARTS) {
                // a part of K: the 16-token chunks are dealt out to the tile's parts; this one's own go into the ring, which is
                // free (all MMAs are done), the others' are parked, [chunk][token][128 rows]
#pragma unroll
                for (int ch = 0; ch < CH; ++ch)
                    if (ch < nch) {
                        const int cc = half * nch + ch;
                        if (cc >= own0 && cc < own1) {
                            float* to = reinterpret_cast<float*>(ring) + (cc - own0) * (16 * TILE_N) + q * 32 + lane;
#pragma unroll
                            for (int e = 0; e < 16; ++e) to[e * TILE_N] = acc[ch * 16 + e];
                        } else {
                            float* to = p.partial + ((size_t)blockIdx.x * chunks + cc) * (16 * TILE_N) + q * 32 + lane;
#pragma unroll
                            for (int e = 0; e < 16; ++e) __stcg(to + e * TILE_N, acc[ch * 16 + e]);
                        }
                    }
                __syncwarp();
                if (lane < p.pk && lane != kpart) red_release_gpu(&p.tickets[2 * (pair - kpart + lane) + rank], 1u);
                if (et == 0) {
                    const unsigned want = 8u * (unsigned)(p.pk - 1);
                    int spins = 0;
#pragma unroll 1
                    while (ld_acquire_gpu(&p.tickets[2 * pair + rank]) < want)
                        if (++spins > SPIN_LIMIT || *abort_flag) { *abort_flag = 1; break; }
                    p.tickets[2 * pair + rank] = 0u;          // ready for the next launch, if everyone has arrived (clear_words)
                    __threadfence();
                }
                asm volatile("bar.sync 1, 256;" ::: "memory");    // (the tile's scale factors are written as well)
            } else {
                asm volatile("bar.sync 1, 256;" ::: "memory");    // the tile's scale factors are written
            }
            // ---- finish, 16 tokens at a time, each warp for itself: its 32 weight rows x 16 tokens go through its own
            //      staging so that a lane then holds 4 neighbouring rows of a token, 8 lanes a token's whole 128 bytes.
            //      (Staged by four warps for 128 rows, a chunk waited at two barriers: T5-xxl-shaped source of
            //      256 tokens 7.5 ms, 6.8 so.)
            const bool scaled = p.ssq_in != nullptr;
            const int c = (lane & 7) * 4, e0 = lane >> 3;     // this lane's rows of the warp's 32, first of its tokens (every 4th)
            const int n = row_tile * OUT_ROWS + rank * (OUT_ROWS / 2) + (MIXED ? q & 1 : q) * 32 + c;
            const int have = min(4, p.N - n);                 // weight rows of this lane inside the matrix
            const bool vec = have == 4 && p.vec_y, add = MODE == 0 && p.epilogue == EPI_ADD;
            float gain[4] = {1.f, 1.f, 1.f, 1.f};
            if (p.out_xs && p.out_gain) {
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    if (j < have) gain[j] = __bfloat162float(p.out_gain[n + j]);
            }
            float* Y = p.Y ? p.Y + n : nullptr;
            // chunks this warp finishes: its half's, or every other one of its part's
            const int ch_end = cut ? own1 - own0 : nch, ch_step = cut ? 2 : 1, ch0 = cut ? half : 0;
            auto column = [&](int ch) { return cut ? (own0 + ch) * 16 : half * htok + ch * 16; };   // in the tile
            float old[4][4];                                  // residual values of a chunk, requested a chunk ahead
            auto load_old = [&](int ch) {
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const int r = tok0 + column(ch) + 4 * k + e0;
                    old[k][0] = old[k][1] = old[k][2] = old[k][3] = 0.f;
                    if (add && ch < ch_end && r < m) {
                        const float* y = Y + (size_t)r * p.ldy;
                        if (vec) {
                            const float4 v = __ldcg(reinterpret_cast<const float4*>(y));
                            old[k][0] = v.x; old[k][1] = v.y; old[k][2] = v.z; old[k][3] = v.w;
                        } else {
#pragma unroll
                            for (int j = 0; j < 4; ++j)
                                if (j < have) old[k][j] = __ldcg(y + j);
                        }
                    }
                }
            };
            load_old(ch0);
            // (mixed: warps q and q + 2 hold gate and up of the same outputs; each finishes half of the chunk's tokens from
            //  both stagings, of which there are two in turn, so that one barrier of the two warps per chunk will do)
            float* buf = staging + ew * ((MIXED ? 2 : NT) * 16 * 32);
            const float* gate = staging + (half * 4 + (q & 1)) * (2 * 16 * 32);
            constexpr int KC = MIXED ? 2 : 4;                 // tokens of a chunk that a lane finishes
            const int k0 = MIXED ? (q >> 1) * 2 : 0;
            float* sums = staging + 8 * 16 * 32;              // [quadrant][token]: sums of squares over a warp's 32 rows
#pragma unroll 1
            for (int ch = ch0; ch < ch_end; ch += ch_step) {
                const int c0 = column(ch), r0 = tok0 + c0;    // column in the tile, token
                if (r0 >= m) break;                           // (the same for the four warps of a half)
                float* put = buf + lane + (MIXED ? (ch & 1) * (16 * 32) : 0);
                // Registers have no index: one short copy per chunk, everything else is a loop over the chunks.  Unrolled
                // over the chunks (100 KB of instructions, pushed out of the caches by the weight stream before every
                // use) it ran at the speed of instruction fetch: up to 3 us a chunk, all SMs in step, against 1 us.
                if (!MIXED) __syncwarp();                     // the chunk before has been read
#define WG_PUT(C)                                                                                                       \
    case C:                                                                                                             \
        if (C < CH) {                                                                                                   \
            _Pragma("unroll") for (int e = 0; e < 16; ++e) {                                                            \
                put[e * 32] = acc[(C < CH ? C : 0) * 16 + e];                                                           \
                if (DUAL) put[(16 + e) * 32] = acc[((NT - 1) * CH + (C < CH ? C : 0)) * 16 + e];                        \
            }                                                                                                           \
        }                                                                                                               \
        break;
                if (!cut) switch (ch) { WG_PUT(0) WG_PUT(1) WG_PUT(2) WG_PUT(3) WG_PUT(4) WG_PUT(5) WG_PUT(6) WG_PUT(7) }
#undef WG_PUT
                if (MIXED) asm volatile("bar.sync %0, 64;" ::"r"(4 + half * 2 + (q & 1)) : "memory");
                else __syncwarp();
                float x[4][4];
                if (cut) {                                    // the parts in order, this one's from the ring
#pragma unroll
                    for (int k = 0; k < 4; ++k) x[k][0] = x[k][1] = x[k][2] = x[k][3] = 0.f;
#pragma unroll 2
                    for (int j = 0; j < p.pk; ++j) {
                        const int at = e0 * TILE_N + q * 32 + c;
                        const float* own = reinterpret_cast<const float*>(ring) + ch * (16 * TILE_N) + at;
                        const float* part = p.partial + ((size_t)(2 * (pair - kpart + j) + rank) * chunks + own0 + ch) * (16 * TILE_N) + at;
                        float4 v[4];
#pragma unroll
                        for (int k = 0; k < 4; ++k)
                            v[k] = j == kpart ? *reinterpret_cast<const float4*>(own + 4 * k * TILE_N) : __ldcg(reinterpret_cast<const float4*>(part + 4 * k * TILE_N));
#pragma unroll
                        for (int k = 0; k < 4; ++k) { x[k][0] += v[k].x; x[k][1] += v[k].y; x[k][2] += v[k].z; x[k][3] += v[k].w; }
                    }
                }
#pragma unroll
                for (int k = 0; k < KC; ++k) {
                    const int e = 4 * (k0 + k) + e0;
                    const float* from = MIXED ? gate + (ch & 1) * (16 * 32) : buf;
                    const float4 v = cut ? make_float4(x[k][0], x[k][1], x[k][2], x[k][3]) : *reinterpret_cast<const float4*>(from + e * 32 + c);
                    const float sc = scaled ? ctl->scale[c0 + e] : 1.f;
                    x[k][0] = v.x * sc; x[k][1] = v.y * sc; x[k][2] = v.z * sc; x[k][3] = v.w * sc;
                    if (DUAL || MIXED) {
                        const float4 u4 = *reinterpret_cast<const float4*>(from + (MIXED ? 2 * 2 * 16 + e : 16 + e) * 32 + c);
                        const float u[4] = {u4.x, u4.y, u4.z, u4.w};
#pragma unroll
                        for (int j = 0; j < 4; ++j)
                            x[k][j] = (p.epilogue == EPI_GEGLU ? gelu_tanh(x[k][j]) : silu(x[k][j])) * (u[j] * sc);
                    }
#pragma unroll
                    for (int j = 0; j < 4; ++j)
                        if (MODE == 0) x[k][j] += old[k][j];
                }
                if (add) load_old(ch + ch_step);
                if (MODE == 0 && p.out_ssq) {                     // (rows past the matrix came out as zeros)
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        float sq = (x[k][0] * x[k][0] + x[k][1] * x[k][1]) + (x[k][2] * x[k][2] + x[k][3] * x[k][3]);
#pragma unroll
                        for (int o = 1; o < 8; o <<= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
                        if ((lane & 7) == 0) sums[q * WG_SET + c0 + 4 * k + e0] = sq;
                    }
                }
#pragma unroll
                for (int k = 0; k < KC; ++k) {
                    const int r = r0 + 4 * (k0 + k) + e0;
                    if (r >= m) continue;
                    if (Y) {
                        float* y = Y + (size_t)r * p.ldy;
                        if (vec) *reinterpret_cast<float4*>(y) = make_float4(x[k][0], x[k][1], x[k][2], x[k][3]);
                        else {
#pragma unroll
                            for (int j = 0; j < 4; ++j)
                                if (j < have) y[j] = x[k][j];
                        }
                    }
                    if (p.out_xs && have > 0) {
                        uint16_t h[4], l[4];
#pragma unroll
                        for (int j = 0; j < 4; ++j) split2f(x[k][j] * gain[j], h[j], l[j]);
                        uint16_t* oh = reinterpret_cast<uint16_t*>(p.out_xs) + (size_t)r * p.out_ld + n;
                        uint16_t* ol = oh + (size_t)p.mpad * p.out_ld;
                        if (have == 4 && (p.out_ld & 3) == 0) {
                            *reinterpret_cast<uint2*>(oh) = make_uint2(h[0] | ((uint32_t)h[1] << 16), h[2] | ((uint32_t)h[3] << 16));
                            *reinterpret_cast<uint2*>(ol) = make_uint2(l[0] | ((uint32_t)l[1] << 16), l[2] | ((uint32_t)l[3] << 16));
                        } else {
#pragma unroll
                            for (int j = 0; j < 4; ++j)
                                if (j < have) { oh[j] = h[j]; ol[j] = l[j]; }
                        }
                    }
                }
            }
            if (MODE == 0 && p.out_ssq) {                         // one piece per token and CTA: its 128 rows
                asm volatile("bar.sync %0, 128;" ::"r"(2 + half) : "memory");
                const int i0 = et & 127, col = (cut ? own0 * 16 : half * htok) + i0;
                if ((cut ? i0 < (own1 - own0) * 16 && ((i0 >> 4) & 1) == half : i0 < htok) && tok0 + col < m)
                    p.out_ssq[(size_t)(row_tile * 2 + rank) * m + tok0 + col] =
                        (sums[col] + sums[WG_SET + col]) + (sums[2 * WG_SET + col] + sums[3 * WG_SET + col]);
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (*abort_flag) {              // (looked at behind the barrier: any warp may have given up last)
        if (tid == 0) set_status(p.status, CSD_ERR_TIMEOUT);
        __nanosleep(2000000);
    }
    cluster_barrier();               // neither CTA leaves while the other's MMAs or arrivals may reach it
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"((uint32_t)(2 * WG_SET)) : "memory");
    }
}

// fp32 rows (times an optional gain) -> two bf16 terms [2][mpad][K] (rows m..mpad-1 zero), plus the
// pieces of each row's sum of squares.  grid = (K / 1024 rounded up, mpad).
__global__ void __launch_bounds__(128)
split2_rows_kernel(const float* __restrict__ X, int ldx, int K, int m, int mpad, const __nv_bfloat16* __restrict__ gain,
                   __nv_bfloat16* __restrict__ xs, float* __restrict__ ssq, unsigned* __restrict__ clear, int clear_count) {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    clear_words(clear, clear_count);
    const int r = blockIdx.y, k = (blockIdx.x * 128 + threadIdx.x) * 8;
    float sq = 0.f;
    if (k < K) {
        float v[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        if (r < m) {
            const float* src = X + (size_t)r * ldx + k;
            const float4 a = *reinterpret_cast<const float4*>(src), b = *reinterpret_cast<const float4*>(src + 4);
            v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w; v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
        }
#pragma unroll
        for (int e = 0; e < 8; ++e) sq = fmaf(v[e], v[e], sq);
        if (gain) {
            const uint4 g = *reinterpret_cast<const uint4*>(gain + k);
            v[0] *= bf16lo(g.x); v[1] *= bf16hi(g.x); v[2] *= bf16lo(g.y); v[3] *= bf16hi(g.y);
            v[4] *= bf16lo(g.z); v[5] *= bf16hi(g.z); v[6] *= bf16lo(g.w); v[7] *= bf16hi(g.w);
        }
        uint32_t t[2][4];
#pragma unroll
        for (int e = 0; e < 8; e += 2) {
            uint16_t a1, a2, c1, c2;
            split2f(v[e], a1, a2);
            split2f(v[e + 1], c1, c2);
            t[0][e / 2] = a1 | ((uint32_t)c1 << 16); t[1][e / 2] = a2 | ((uint32_t)c2 << 16);
        }
#pragma unroll
        for (int s = 0; s < 2; ++s)
            *reinterpret_cast<uint4*>(xs + (size_t)(s * mpad + r) * K + k) = make_uint4(t[s][0], t[s][1], t[s][2], t[s][3]);
    }
    __shared__ float part[4];
    sq = warp_sum(sq);
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = sq;
    __syncthreads();
    if (threadIdx.x == 0 && ssq && r < m) ssq[(size_t)blockIdx.x * m + r] = (part[0] + part[1]) + (part[2] + part[3]);
}

csd_status launch_wide_split(const float* X, int ldx, int K, int m, const __nv_bfloat16* gain, __nv_bfloat16* xs,
                             float* ssq, cudaStream_t st, unsigned* clear, int clear_count) {
    if (!X || !xs || (((uintptr_t)X) & 15) || (ldx & 3) || (K & 7) || m < 1 || m > CSD_WIDE_ROWS) return CSD_ERR_INVALID_ARG;
    const int mpad = (m + 15) & ~15;
    PdlLaunch L(dim3((unsigned)wide_split_pieces(K), (unsigned)mpad), dim3(128), 0, st);
    CSD_CUDA(cudaLaunchKernelEx(&L.cfg, split2_rows_kernel, X, ldx, K, m, mpad, gain, xs, ssq, clear, clear_count));
    count_launch();
    return CSD_OK;
}

template <int MODE, bool MERGED, bool PARTS = false>
static csd_status launch_wg(const CUtensorMap& tw, const CUtensorMap& tw2, const CUtensorMap& tx, const WgParams& wp,
                            const WgPlan& pl, cudaStream_t st) {
    auto kern = wide_gemm_kernel<MODE, MERGED, PARTS>;
    static PerDevice ready;
    const csd_status ok = allow_smem(ready, kern, WG_SMEM_MAX);
    if (ok != CSD_OK) return ok;
    cudaLaunchConfig_t cfg = cudaLaunchConfig_t{};
    cudaLaunchAttribute attr[2];
    cfg.gridDim = dim3((unsigned)(2 * pl.pairs)); cfg.blockDim = dim3(WG_THREADS); cfg.dynamicSmemBytes = pl.smem; cfg.stream = st;
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = 2; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr; cfg.numAttrs = 2;
    CSD_CUDA(cudaLaunchKernelEx(&cfg, kern, tw, tw2, tx, wp));
    count_launch();
    return CSD_OK;
}

csd_status launch_linear_wide(const WideArgs& a, cudaStream_t st) {
    const bool dual = a.W2 != nullptr;
    if (!a.W || !a.xs || (((uintptr_t)a.xs) & 15) || !a.partial || !a.tickets) return CSD_ERR_INVALID_ARG;
    if (!a.Y && (!dual || !a.out_xs)) return CSD_ERR_INVALID_ARG;
    if (dual != (a.epilogue == EPI_SWIGLU || a.epilogue == EPI_GEGLU) || (dual && a.out_ssq)) return CSD_ERR_INVALID_ARG;
    if (!wide_supported(a.m, a.N, a.K, dual)) return CSD_ERR_UNSUPPORTED;
    const WgPlan pl = wg_plan(a.m, a.N, a.K, dual);
    CUtensorMap tw, tw2, tx;
    const int box = pl.mixed ? TILE_N / 2 : TILE_N;
    if (!tensor_map_2d(a.W, a.N, a.K, box, &tw)) return CSD_ERR_UNSUPPORTED;
    tw2 = tw;
    if (dual && !tensor_map_2d(a.W2, a.N, a.K, box, &tw2)) return CSD_ERR_UNSUPPORTED;
    if (!tensor_map_2d(a.xs, 2 * pl.mpad, a.K, pl.merged ? pl.nt : pl.nt / 2, &tx)) return CSD_ERR_UNSUPPORTED;
    WgParams wp;
    wp.Y = a.Y; wp.partial = a.partial; wp.tickets = a.tickets; wp.status = status_word_device();
    wp.ssq_in = a.ssq; wp.ssq_cnt = a.ssq_cnt;
    wp.out_xs = a.out_xs; wp.out_gain = a.out_gain; wp.out_ssq = a.out_ssq; wp.out_ld = a.out_ld;
    wp.m = a.m; wp.mpad = pl.mpad; wp.nt = pl.nt; wp.ntok = pl.ntok; wp.tiles = pl.tiles; wp.nkb = pl.nkb; wp.pk = pl.pk;
    wp.gran = pl.gran; wp.N = a.N; wp.K = a.K; wp.ldy = a.ldy; wp.stages = pl.stages; wp.epilogue = a.epilogue; wp.eps = a.eps;
    wp.vec_y = (a.ldy & 3) == 0 && (((uintptr_t)a.Y) & 15) == 0;
    if (dual && !pl.mixed) return launch_wg<1, true>(tw, tw2, tx, wp, pl, st);
    if (dual) return pl.merged ? launch_wg<2, true>(tw, tw2, tx, wp, pl, st) : launch_wg<2, false>(tw, tw2, tx, wp, pl, st);
    if (pl.pk > 1) return pl.merged ? launch_wg<0, true, true>(tw, tw2, tx, wp, pl, st) : launch_wg<0, false, true>(tw, tw2, tx, wp, pl, st);
    return pl.merged ? launch_wg<0, true>(tw, tw2, tx, wp, pl, st) : launch_wg<0, false>(tw, tw2, tx, wp, pl, st);
}

}  // namespace csd
