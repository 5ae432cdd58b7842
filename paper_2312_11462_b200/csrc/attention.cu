// Attention of a block of m <= 17 query rows against a bf16 K/V cache, split along the keys.
//
// grid = (heads, splits), the splits of one head forming a thread-block cluster.  A CTA walks its
// key range in tiles of 64 positions: thread 0 requests each tile's committed rows with two bulk
// copies (a head's rows are contiguous in the cache) that complete on an mbarrier, two tiles in
// flight; the block's own rows (self-attention of a drafted block) are rotated, rounded to bf16,
// written to the cache and laid over the staged tile by the CTA whose range holds them, so the
// separate append pass and its round trip through HBM are gone.  Every CTA keeps an online softmax
// per row (running max, running sum, rescaled accumulator); the splits then exchange (max, sum,
// unnormalised output) through distributed shared memory and each merges a slice of the output.
// Rows see keys [0, n_keys + r) when causal, all n_keys otherwise (cross-attention, encoder).
#include <cooperative_groups.h>
#include "attention.cuh"
#include "attention_mma.cuh"
#include "gemm_tc.cuh"

namespace cg = cooperative_groups;

namespace csd {

constexpr int AT = 256;
constexpr int MAXM = CSD_MAX_ROWS;
constexpr int MAX_SPLITS = 8;          // portable cluster size
constexpr int STAGES = 2;

template <int DH> struct AttnCfg {
    static constexpr int HP = DH / 2;                        // dim pairs
    static constexpr int G = AT / HP;                        // row groups in the PV phase
    static constexpr int RG = (MAXM + G - 1) / G;            // rows per group
    static constexpr int NC = DH / 32;                       // 8-element chunks per score thread
    static constexpr int QROW = NC * 36;                     // q row: 32-float groups, 4 floats of skew each
    static constexpr int REC = DH + 4;                       // merge record: output row, max, sum (and 16-byte rows)
    static constexpr size_t TILE_BYTES = (size_t)TILE * DH * 2;
    static constexpr size_t QS_FLOATS = (size_t)MAXM * (QROW > REC ? QROW : REC);
    static constexpr size_t SMEM = 2 * STAGES * TILE_BYTES + QS_FLOATS * 4 + (size_t)MAXM * TILE * 4 +
                                   2 * (size_t)MAXM * DH * 2 + 3 * 32 * 4 + 128;
};

struct AttnParams {
    const float* q; const float* k_new; const float* v_new; const float* rope_cos; const float* rope_sin;
    __nv_bfloat16* Kc; __nv_bfloat16* Vc; const float* bias; float* out;
    __nv_bfloat16* out_xs; int out_xs_ld;
    int xs_m, xs_r0;        // three-term output: rows per term of the whole buffer, row of this block's first row
    int* status;
    int ldq, ld_new, m, cap, H, n_keys, n_old, early_loads, causal, bias_len, bias_zero, q_pos0, ldo, nsplit, split_len;
    float scale;
    // tree-shaped block: row r sees block row j only if bit j of tmask[r] is set (its ancestors and
    // itself) and is rotated for position n_old + tdepth[r]; its cache slot stays n_old + r
    int tree;
    unsigned tmask[MAXM];
    unsigned char tdepth[MAXM];
};

// What differs between the sequences of a batched review: grid.z of the tensor-core kernel picks one.  (A launch per
// sequence: three blocks of 5, 3 and 5 rows of the 7B shape 3569 us, 3347 so.)
constexpr int MAX_SEGS = 4;
struct AttnSeg {
    const float* q; const float* k_new; const float* v_new; __nv_bfloat16* Kc; __nv_bfloat16* Vc; float* out;
    int m, n_keys, n_old, split_len, q_pos0, xs_r0;
};
struct AttnSegs { CUtensorMap k[MAX_SEGS], v[MAX_SEGS]; AttnSeg seg[MAX_SEGS]; };

__device__ __forceinline__ void bulk_load(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(smem_u32(dst)), "l"(src), "r"(bytes), "r"(smem_u32(bar)) : "memory");
}

// two neighbouring output columns of row r as three bf16 terms each (rows term * m + r)
__device__ __forceinline__ void store_split(__nv_bfloat16* xs, int ld, int m, int r, int col, float a, float b) {
    uint16_t a1, a2, a3, c1, c2, c3;
    split3(a, a1, a2, a3);
    split3(b, c1, c2, c3);
    uint32_t* base = reinterpret_cast<uint32_t*>(reinterpret_cast<uint16_t*>(xs) + col);
    base[((size_t)r * ld) >> 1] = a1 | ((uint32_t)c1 << 16);
    base[((size_t)(m + r) * ld) >> 1] = a2 | ((uint32_t)c2 << 16);
    base[((size_t)(2 * m + r) * ld) >> 1] = a3 | ((uint32_t)c3 << 16);
}

// W neighbouring values
__device__ __forceinline__ void load_vec(const float* p, float (&v)[1]) { v[0] = *p; }
__device__ __forceinline__ void load_vec(const float* p, float (&v)[2]) {
    const float2 f = *reinterpret_cast<const float2*>(p);
    v[0] = f.x; v[1] = f.y;
}
__device__ __forceinline__ void load_vec(const float* p, float (&v)[4]) {
    const float4 f = *reinterpret_cast<const float4*>(p);
    v[0] = f.x; v[1] = f.y; v[2] = f.z; v[3] = f.w;
}
__device__ __forceinline__ void store_words(void* p, const uint32_t (&w)[1]) { *reinterpret_cast<uint32_t*>(p) = w[0]; }
__device__ __forceinline__ void store_words(void* p, const uint32_t (&w)[2]) { *reinterpret_cast<uint2*>(p) = make_uint2(w[0], w[1]); }

// Merge of the splits' records (unnormalised output row, running max, running sum) through
// distributed shared memory: the CTAs of a head share out the m*DH output elements, W neighbours a thread; each thread
// first fetches everything it needs from all splits in one batch of independent remote loads.
template <int DH, int REC, int W>
__device__ __forceinline__ void merge_rows(cg::cluster_group& cluster, float* rec, const AttnParams& p, float* out, int xs_r0,
                                             int h, int split, int m) {
    for (int i = split * AT + threadIdx.x; i < m * (DH / W); i += p.nsplit * AT) {
        const int r = i / (DH / W), d = i % (DH / W) * W;
        float ms[MAX_SPLITS], ls[MAX_SPLITS], vs[MAX_SPLITS][W];
#pragma unroll
        for (int s = 0; s < MAX_SPLITS; ++s) {
            ms[s] = -INFINITY; ls[s] = 0.f;
#pragma unroll
            for (int w = 0; w < W; ++w) vs[s][w] = 0.f;
            if (s < p.nsplit) {
                const float* rs = cluster.map_shared_rank(rec, s) + r * REC;
                ms[s] = rs[DH]; ls[s] = rs[DH + 1];
                load_vec(rs + d, vs[s]);
            }
        }
        float M = -INFINITY;
#pragma unroll
        for (int s = 0; s < MAX_SPLITS; ++s) M = fmaxf(M, ms[s]);
        float num[W], den = 0.f;
#pragma unroll
        for (int w = 0; w < W; ++w) num[w] = 0.f;
#pragma unroll
        for (int s = 0; s < MAX_SPLITS; ++s)
            if (ms[s] > -INFINITY) {
                const float f = expf(ms[s] - M);
#pragma unroll
                for (int w = 0; w < W; ++w) num[w] = fmaf(vs[s][w], f, num[w]);
                den = fmaf(ls[s], f, den);
            }
        float ov[W];
        uint16_t b[3][W];
#pragma unroll
        for (int w = 0; w < W; ++w) {
            ov[w] = den > 0.f ? num[w] / den : 0.f;
            split3(ov[w], b[0][w], b[1][w], b[2][w]);
        }
        if (p.out_xs) {
#pragma unroll
            for (int t = 0; t < 3; ++t) {
                __nv_bfloat16* dst = p.out_xs + (size_t)(t * p.xs_m + xs_r0 + r) * p.out_xs_ld + h * DH + d;
                if constexpr (W == 1) {
                    *reinterpret_cast<uint16_t*>(dst) = b[t][0];
                } else {
                    uint32_t w2[W / 2];
#pragma unroll
                    for (int w = 0; w < W; w += 2) w2[w / 2] = b[t][w] | ((uint32_t)b[t][w + 1] << 16);
                    store_words(dst, w2);
                }
            }
        } else {
#pragma unroll
            for (int w = 0; w < W; ++w) out[(size_t)r * p.ldo + h * DH + d + w] = ov[w];
        }
    }
}
// one element a thread while there are threads for all, four otherwise
template <int DH, int REC>
__device__ __forceinline__ void merge_splits(cg::cluster_group& cluster, float* rec, const AttnParams& p, float* out, int xs_r0,
                                             int h, int split, int m) {
    if (m * DH <= p.nsplit * AT) merge_rows<DH, REC, 1>(cluster, rec, p, out, xs_r0, h, split, m);
    else merge_rows<DH, REC, 4>(cluster, rec, p, out, xs_r0, h, split, m);
}

template <int DH>
__global__ void __launch_bounds__(AT)
block_attention_kernel(const AttnParams p) {
    using C = AttnCfg<DH>;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    __nv_bfloat16* Ks = reinterpret_cast<__nv_bfloat16*>(smem_raw);            // [STAGES][TILE][DH]
    __nv_bfloat16* Vs = Ks + STAGES * TILE * DH;
    float* qs = reinterpret_cast<float*>(Vs + STAGES * TILE * DH);            // [MAXM][QROW]; later [MAXM][REC]
    float* sc = qs + C::QS_FLOATS;                                            // [MAXM][TILE]
    __nv_bfloat16* newK = reinterpret_cast<__nv_bfloat16*>(sc + MAXM * TILE); // [MAXM][DH] the block's own rows
    __nv_bfloat16* newV = newK + MAXM * DH;
    float* row_m = reinterpret_cast<float*>(newV + MAXM * DH);                // [32]
    float* row_l = row_m + 32;
    float* row_a = row_l + 32;
    uint64_t* full = reinterpret_cast<uint64_t*>(row_a + 32);                 // [STAGES]

    cg::cluster_group cluster = cg::this_cluster();
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int h = blockIdx.x, split = blockIdx.y;
    const int m = p.m, half = DH / 2;
    const int total = p.causal ? p.n_keys + m - 1 : p.n_keys;   // keys any row may see
    const int s_begin = split * p.split_len;
    const int s_end = min(total, s_begin + p.split_len);
    const int n_tiles = s_end > s_begin ? (s_end - s_begin + TILE - 1) / TILE : 0;
    __nv_bfloat16* Kh = p.Kc + (size_t)h * p.cap * DH;
    __nv_bfloat16* Vh = p.Vc + (size_t)h * p.cap * DH;
    const float* bias_h = p.bias ? p.bias + (size_t)h * p.bias_len : nullptr;

    if (tid == 0) {
        for (int s = 0; s < STAGES; ++s) mbar_init(&full[s], 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (tid < 32) { row_m[tid] = -INFINITY; row_l[tid] = 0.f; row_a[tid] = 1.f; }
    __syncthreads();


    // committed rows of tile `it` (the rest of the tile, if any, are the block's own rows)
    auto old_rows = [&](int it) {
        const int t0 = s_begin + it * TILE;
        return max(0, min(min(t0 + TILE, s_end), p.n_old) - t0);
    };
    auto request = [&](int it) {
        const int st = it % STAGES, t0 = s_begin + it * TILE, cnt = old_rows(it);
        if (cnt <= 0) return;
        const uint32_t bytes = (uint32_t)cnt * DH * 2;
        mbar_expect_tx(&full[st], 2 * bytes);
        bulk_load(Ks + (size_t)st * TILE * DH, Kh + (size_t)t0 * DH, bytes, &full[st]);
        bulk_load(Vs + (size_t)st * TILE * DH, Vh + (size_t)t0 * DH, bytes, &full[st]);
    };
    // Committed rows were written by the attention kernel of an earlier forward; between that
    // kernel and this one the stream holds at least one kernel that waits for its predecessor
    // before it lets its successor start, so those rows are complete and may be requested before
    // this kernel's own dependency wait.  q and the block's k and v rows come from the kernel
    // right before this one.  The encoder's self-attention reads rows the previous kernel wrote:
    // there the requests wait too.
    if (tid == 0 && p.early_loads)
        for (int it = 0; it < n_tiles && it < STAGES; ++it) request(it);
    pdl_wait();
    pdl_trigger();
    if (tid == 0 && !p.early_loads)
        for (int it = 0; it < n_tiles && it < STAGES; ++it) request(it);

    // ---- the block's rows: q (rotated) into shared memory; k (rotated) and v rounded to bf16, kept
    //      for the tiles that hold them and written to the cache by the CTA whose range they fall in
    for (int i = tid; i < m * half; i += AT) {
        const int r = i / half, d = i % half, pos = p.n_old + r;
        const int rpos = p.n_old + (p.tree ? (int)p.tdepth[r] : r);      // position the rotation uses
        float c = 1.f, s = 0.f;
        if (p.rope_cos) { c = p.rope_cos[(size_t)rpos * half + d]; s = p.rope_sin[(size_t)rpos * half + d]; }
        const float* qr = p.q + (size_t)r * p.ldq + h * DH;
        const float q0 = qr[d], q1 = qr[d + half];
        const int e0 = d, e1 = d + half;
        qs[r * C::QROW + (e0 >> 5) * 36 + (e0 & 31)] = q0 * c - q1 * s;
        qs[r * C::QROW + (e1 >> 5) * 36 + (e1 & 31)] = q0 * s + q1 * c;
        if (p.k_new) {
            const float* kr = p.k_new + (size_t)r * p.ld_new + h * DH;
            const float* vr = p.v_new + (size_t)r * p.ld_new + h * DH;
            const float k0 = kr[d], k1 = kr[d + half];
            const __nv_bfloat16 ka = __float2bfloat16_rn(k0 * c - k1 * s), kb = __float2bfloat16_rn(k0 * s + k1 * c);
            const __nv_bfloat16 va = __float2bfloat16_rn(vr[d]), vb = __float2bfloat16_rn(vr[d + half]);
            newK[r * DH + d] = ka; newK[r * DH + d + half] = kb;
            newV[r * DH + d] = va; newV[r * DH + d + half] = vb;
            if (pos >= s_begin && pos < s_end) {
                Kh[(size_t)pos * DH + d] = ka; Kh[(size_t)pos * DH + d + half] = kb;
                Vh[(size_t)pos * DH + d] = va; Vh[(size_t)pos * DH + d + half] = vb;
            }
        }
    }

    const int dp = tid % C::HP, g = tid / C::HP;
    float acc[C::RG][2];
#pragma unroll
    for (int rr = 0; rr < C::RG; ++rr) { acc[rr][0] = 0.f; acc[rr][1] = 0.f; }

    bool failed = false;
    for (int it = 0; it < n_tiles; ++it) {
        const int st = it % STAGES, t0 = s_begin + it * TILE;
        const int ok = old_rows(it) <= 0 || mbar_wait(&full[st], (uint32_t)(it / STAGES) & 1u);
        if (__syncthreads_or(!ok)) {      // (also orders the set-up above before the first tile)
            if (!ok) mbar_wait(&full[st], (uint32_t)(it / STAGES) & 1u);   // once more, so no copy is in flight at exit
            failed = true;
            break;
        }
        __nv_bfloat16* Kt = Ks + (size_t)st * TILE * DH;
        __nv_bfloat16* Vt = Vs + (size_t)st * TILE * DH;
        const int valid = min(TILE, s_end - t0);
        {   // lay the block's own rows over the tile; clear the value rows past the end of the range
            const int new_lo = max(t0, p.n_old), n_new = t0 + valid - new_lo;
            for (int idx = tid; idx < n_new * (DH / 8); idx += AT) {
                const int row = idx / (DH / 8), c = idx % (DH / 8), j = new_lo + row - t0, r = new_lo + row - p.n_old;
                *reinterpret_cast<uint4*>(Kt + j * DH + c * 8) = *reinterpret_cast<const uint4*>(newK + r * DH + c * 8);
                *reinterpret_cast<uint4*>(Vt + j * DH + c * 8) = *reinterpret_cast<const uint4*>(newV + r * DH + c * 8);
            }
            for (int idx = tid; idx < (TILE - valid) * (DH / 8); idx += AT)
                *reinterpret_cast<uint4*>(Vt + (size_t)valid * DH + idx * 8) = make_uint4(0, 0, 0, 0);
        }
        __syncthreads();
        // ---- scores: 4 threads per key, each over a quarter of the head dimension.  The 32-element
        //      group a thread reads at step c is rotated by the key index, so that neighbouring keys
        //      (whose rows start a multiple of 128 bytes apart) hit different banks.
        {
            const int j = tid >> 2, part = tid & 3;
            uint4 kreg[C::NC];
#pragma unroll
            for (int c = 0; c < C::NC; ++c)
                kreg[c] = *reinterpret_cast<const uint4*>(Kt + j * DH + (((c + j) % C::NC) * 4 + part) * 8);
            const int key = t0 + j;
            for (int r = 0; r < m; ++r) {
                float d = 0.f;
#pragma unroll
                for (int c = 0; c < C::NC; ++c) {
                    const float* qp = qs + r * C::QROW + ((c + j) % C::NC) * 36 + part * 8;
                    const float4 qa = *reinterpret_cast<const float4*>(qp);
                    const float4 qb = *reinterpret_cast<const float4*>(qp + 4);
                    d = fmaf(bf16lo(kreg[c].x), qa.x, d); d = fmaf(bf16hi(kreg[c].x), qa.y, d);
                    d = fmaf(bf16lo(kreg[c].y), qa.z, d); d = fmaf(bf16hi(kreg[c].y), qa.w, d);
                    d = fmaf(bf16lo(kreg[c].z), qb.x, d); d = fmaf(bf16hi(kreg[c].z), qb.y, d);
                    d = fmaf(bf16lo(kreg[c].w), qb.z, d); d = fmaf(bf16hi(kreg[c].w), qb.w, d);
                }
                d += __shfl_xor_sync(0xffffffffu, d, 1);
                d += __shfl_xor_sync(0xffffffffu, d, 2);
                if (part == 0) {
                    const int limit = p.causal ? p.n_keys + r : p.n_keys;   // keys [0, limit)
                    float s = -INFINITY;
                    bool vis = key < s_end && key < limit;
                    if (p.tree && key >= p.n_old) vis = key < s_end && ((p.tmask[r] >> (key - p.n_old)) & 1u);
                    if (vis) {
                        s = d * p.scale;
                        if (bias_h) {
                            int bi = key - (p.q_pos0 + r) + p.bias_zero;
                            bi = max(0, min(p.bias_len - 1, bi));
                            s += bias_h[bi];
                        }
                    }
                    sc[r * TILE + j] = s;
                }
            }
        }
        __syncthreads();
        // ---- online softmax bookkeeping: warp w owns rows w, w+8, w+16
        for (int r = warp; r < m; r += AT / 32) {
            const float s0 = sc[r * TILE + lane], s1 = sc[r * TILE + lane + 32];
            const float tmax = warp_max(fmaxf(s0, s1));
            const float old = row_m[r];
            const float nm = fmaxf(old, tmax);
            float p0 = 0.f, p1 = 0.f, alpha = 1.f;
            if (nm > -INFINITY) {
                p0 = expf(s0 - nm);
                p1 = expf(s1 - nm);
                alpha = expf(old - nm);
            }
            sc[r * TILE + lane] = p0;
            sc[r * TILE + lane + 32] = p1;
            const float tsum = warp_sum(p0 + p1);
            if (lane == 0) {
                row_m[r] = nm;
                row_l[r] = row_l[r] * alpha + tsum;
                row_a[r] = alpha;
            }
        }
        __syncthreads();
        // ---- P.V: thread owns one dim pair for the rows of its group
#pragma unroll
        for (int rr = 0; rr < C::RG; ++rr) {
            const int r = g + rr * C::G;
            if (r < m) { const float a = row_a[r]; acc[rr][0] *= a; acc[rr][1] *= a; }
        }
        for (int j4 = 0; j4 < TILE; j4 += 4) {
            float v[4][2];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const uint32_t w = *reinterpret_cast<const uint32_t*>(Vt + (j4 + i) * DH + 2 * dp);
                v[i][0] = bf16lo(w); v[i][1] = bf16hi(w);
            }
#pragma unroll
            for (int rr = 0; rr < C::RG; ++rr) {
                const int r = g + rr * C::G;
                if (r < m) {
                    const float4 pp = *reinterpret_cast<const float4*>(sc + r * TILE + j4);
                    acc[rr][0] = fmaf(pp.x, v[0][0], acc[rr][0]); acc[rr][1] = fmaf(pp.x, v[0][1], acc[rr][1]);
                    acc[rr][0] = fmaf(pp.y, v[1][0], acc[rr][0]); acc[rr][1] = fmaf(pp.y, v[1][1], acc[rr][1]);
                    acc[rr][0] = fmaf(pp.z, v[2][0], acc[rr][0]); acc[rr][1] = fmaf(pp.z, v[2][1], acc[rr][1]);
                    acc[rr][0] = fmaf(pp.w, v[3][0], acc[rr][0]); acc[rr][1] = fmaf(pp.w, v[3][1], acc[rr][1]);
                }
            }
        }
        __syncthreads();           // tile consumed: its stage may be filled again
        if (tid == 0 && it + STAGES < n_tiles) {
            fence_async_smem();    // the overlay above wrote this stage through the generic proxy
            request(it + STAGES);
        }
    }
    if (failed && tid == 0) set_status(p.status, CSD_ERR_TIMEOUT);

    if (p.nsplit == 1) {
#pragma unroll
        for (int rr = 0; rr < C::RG; ++rr) {
            const int r = g + rr * C::G;
            if (r < m) {
                const float inv = row_l[r] > 0.f ? 1.f / row_l[r] : 0.f;
                const float a = acc[rr][0] * inv, b = acc[rr][1] * inv;
                if (p.out_xs) store_split(p.out_xs, p.out_xs_ld, p.xs_m, p.xs_r0 + r, h * DH + 2 * dp, a, b);
                else *reinterpret_cast<float2*>(p.out + (size_t)r * p.ldo + h * DH + 2 * dp) = make_float2(a, b);
            }
        }
        return;
    }
    // ---- leave this split's (output, max, sum) in shared memory; after the cluster barrier every
    //      CTA of the head merges its share of the output elements from all the splits' records
    float* rec = qs;      // the q rows are not needed any more (all threads are past the last tile)
#pragma unroll
    for (int rr = 0; rr < C::RG; ++rr) {
        const int r = g + rr * C::G;
        if (r < m) {
            rec[r * C::REC + 2 * dp] = acc[rr][0];
            rec[r * C::REC + 2 * dp + 1] = acc[rr][1];
        }
    }
    if (tid < m) { rec[tid * C::REC + DH] = row_m[tid]; rec[tid * C::REC + DH + 1] = row_l[tid]; }
    cluster.sync();
    merge_splits<DH, C::REC>(cluster, rec, p, p.out, p.xs_r0, h, split, m);
    cluster.sync();       // no CTA leaves while another may still read its record
}

// -------------------------------------------------------------------------------------------------
// Tensor-core variant (head dimension 64 or 128): the same walk over 64-key tiles, with the two
// contractions of a tile on mma.sync (m16n8k16, bf16 operands, fp32 accumulators).  K and V tiles
// arrive by tensor-map TMA copies with the 128-byte swizzle, which makes the ldmatrix reads of
// their rows conflict-free; q and the softmax weights, fp32 quantities, enter the MMAs as a
// bf16 pair (value = hi + lo, two MMAs), so the products keep 16 mantissa bits while K and V,
// bf16 in the cache, are exact.  Warp w owns keys 8w..8w+7 of the tile in q.K^T and output
// dimensions 16w..16w+15 in P.V; rows 16..31 (a 17-row block) are a second m16 tile.
// -------------------------------------------------------------------------------------------------
template <int DH> struct MmaCfg {
    static constexpr int QP = DH * 2 + 16;                   // bytes per q row: bf16 plus one 16-byte skew
    static constexpr int PP = TILE * 2 + 16;                 // bytes per row of softmax weights
    static constexpr int SP = TILE + 4;                      // floats per score row
    static constexpr int REC = DH + 4;
    static constexpr int NBOX = DH / 64;                     // 64-dimension (128-byte) boxes per row
    static constexpr size_t TILE_BYTES = (size_t)TILE * DH * 2;
    static constexpr size_t smem(int rows) {                 // rows = 16 or 32 operand rows
        return 1024 + 2 * STAGES * TILE_BYTES + 2 * (size_t)rows * QP + (size_t)rows * SP * 4 + 2 * (size_t)rows * PP +
               2 * (size_t)MAXM * DH * 2 + 3 * 32 * 4 + 64;
    }
};
template <int DH, int MT>
__global__ void __launch_bounds__(AT)
block_attention_mma_kernel(const __grid_constant__ AttnSegs segs, const AttnParams p) {
    using C = MmaCfg<DH>;
    const AttnSeg& sg = segs.seg[blockIdx.z];
    constexpr int R = MT * 16;
    extern __shared__ unsigned char smem_dyn[];
    unsigned char* base = (unsigned char*)(((uintptr_t)smem_dyn + 1023) & ~(uintptr_t)1023);
    unsigned char* Ks = base;                                        // [STAGES][tile], swizzled
    unsigned char* Vs = Ks + STAGES * C::TILE_BYTES;
    unsigned char* qh = Vs + STAGES * C::TILE_BYTES;                 // [R][QP] high parts of q; later the merge record
    unsigned char* ql = qh + R * C::QP;
    float* sc = reinterpret_cast<float*>(ql + R * C::QP);            // [R][SP]
    unsigned char* ph = reinterpret_cast<unsigned char*>(sc + R * C::SP);   // [R][PP]
    unsigned char* pl = ph + R * C::PP;
    __nv_bfloat16* newK = reinterpret_cast<__nv_bfloat16*>(pl + R * C::PP); // [MAXM][DH]
    __nv_bfloat16* newV = newK + MAXM * DH;
    float* row_m = reinterpret_cast<float*>(newV + MAXM * DH);
    float* row_l = row_m + 32;
    float* row_a = row_l + 32;
    uint64_t* full = reinterpret_cast<uint64_t*>(row_a + 32);

    cg::cluster_group cluster = cg::this_cluster();
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int h = blockIdx.x, split = blockIdx.y;
    const int m = sg.m, half = DH / 2, n_keys = sg.n_keys;
    const int total = p.causal ? n_keys + m - 1 : n_keys;
    const int n_old = sg.n_old;
    const int s_begin = split * sg.split_len;
    const int s_end = min(total, s_begin + sg.split_len);
    const int n_tiles = s_end > s_begin ? (s_end - s_begin + TILE - 1) / TILE : 0;
    __nv_bfloat16* Kh = sg.Kc + (size_t)h * p.cap * DH;
    __nv_bfloat16* Vh = sg.Vc + (size_t)h * p.cap * DH;
    const float* bias_h = p.bias ? p.bias + (size_t)h * p.bias_len : nullptr;

    if (tid == 0) {
        for (int s = 0; s < STAGES; ++s) mbar_init(&full[s], 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (tid < 32) { row_m[tid] = -INFINITY; row_l[tid] = 0.f; row_a[tid] = 1.f; }
    // operand rows past the block stay zero (q, and the softmax weights, which are rewritten per tile only for real rows)
    for (int i = tid; i < (2 * R * C::QP + R * C::SP * 4 + 2 * R * C::PP) / 16; i += AT)
        reinterpret_cast<uint4*>(qh)[i] = make_uint4(0, 0, 0, 0);
    __syncthreads();

    auto request = [&](int it) {       // whole 64-row boxes: rows the block itself supplies are laid over afterwards
        const int st = it % STAGES, row0 = h * p.cap + s_begin + it * TILE;
        mbar_expect_tx(&full[st], 2 * (uint32_t)C::TILE_BYTES);
#pragma unroll
        for (int b = 0; b < C::NBOX; ++b) {
            tma_load_2d(Ks + st * C::TILE_BYTES + b * (TILE * 128), &segs.k[blockIdx.z], &full[st], b * 64, row0);
            tma_load_2d(Vs + st * C::TILE_BYTES + b * (TILE * 128), &segs.v[blockIdx.z], &full[st], b * 64, row0);
        }
    };
    // (see the CUDA-core kernel above for why the requests may precede the dependency wait)
    if (tid == 0 && p.early_loads)
        for (int it = 0; it < n_tiles && it < STAGES; ++it) request(it);
    // this thread's items of the block: W neighbouring rotation pairs of a row each; their factors are constants.  (One element an
    // item cost 17 rows of the 7B shape 3 us a layer more and 12 rows 1.5; four of a one-tile block leave too few threads at work.)
    constexpr int W = MT == 1 ? 2 : 4, PER_ROW = DH / 2 / W, ITEMS = (R * PER_ROW + AT - 1) / AT;
    float rc[ITEMS][W], rs[ITEMS][W];
#pragma unroll
    for (int e = 0; e < ITEMS; ++e) {
        const int i = tid + e * AT, r = i / PER_ROW;
#pragma unroll
        for (int w = 0; w < W; ++w) { rc[e][w] = 1.f; rs[e][w] = 0.f; }
        if (r < m && p.rope_cos) {
            const size_t at = (size_t)(n_old + (p.tree ? (int)p.tdepth[r] : r)) * half + i % PER_ROW * W;
            load_vec(p.rope_cos + at, rc[e]);
            load_vec(p.rope_sin + at, rs[e]);
        }
    }
    pdl_wait();
    pdl_trigger();
    if (tid == 0 && !p.early_loads)
        for (int it = 0; it < n_tiles && it < STAGES; ++it) request(it);

    // ---- the block's rows: q rotated and split into its bf16 pair; k rotated, v, both rounded to bf16 (by the splits whose
    //      range holds some of them).  All loads first (one round trip), then the arithmetic and the stores.
    {
        const bool fresh = sg.k_new && s_end > n_old;
        float q0[ITEMS][W], q1[ITEMS][W], k0[ITEMS][W], k1[ITEMS][W], v0[ITEMS][W], v1[ITEMS][W];
#pragma unroll
        for (int e = 0; e < ITEMS; ++e) {
            const int i = tid + e * AT, r = i / PER_ROW, d = i % PER_ROW * W;
            if (r < m) {
                const float* qr = sg.q + (size_t)r * p.ldq + h * DH + d;
                load_vec(qr, q0[e]);
                load_vec(qr + half, q1[e]);
                if (fresh) {
                    const float* kr = sg.k_new + (size_t)r * p.ld_new + h * DH + d;
                    const float* vr = sg.v_new + (size_t)r * p.ld_new + h * DH + d;
                    load_vec(kr, k0[e]);
                    load_vec(kr + half, k1[e]);
                    load_vec(vr, v0[e]);
                    load_vec(vr + half, v1[e]);
                }
            }
        }
#pragma unroll
        for (int e = 0; e < ITEMS; ++e) {
            const int i = tid + e * AT, r = i / PER_ROW, d = i % PER_ROW * W, pos = n_old + r;
            if (r >= m) continue;
            auto turn = [&](float (&a)[W], float (&b)[W]) {
#pragma unroll
                for (int w = 0; w < W; ++w) {
                    const float x = a[w], y = b[w];
                    a[w] = x * rc[e][w] - y * rs[e][w];
                    b[w] = x * rs[e][w] + y * rc[e][w];
                }
            };
            uint32_t hi[W / 2], lo[W / 2];
            auto put_pair = [&](const float (&v)[W], int col) {
#pragma unroll
                for (int w = 0; w < W; w += 2) pack_pair(v[w], v[w + 1], hi[w / 2], lo[w / 2]);
                store_words(qh + r * C::QP + col * 2, hi);
                store_words(ql + r * C::QP + col * 2, lo);
            };
            turn(q0[e], q1[e]);
            put_pair(q0[e], d);
            put_pair(q1[e], d + half);
            if (fresh) {
                turn(k0[e], k1[e]);
                const bool mine = pos >= s_begin && pos < s_end;
                auto put = [&](const float (&v)[W], __nv_bfloat16* smem, __nv_bfloat16* cache, int col) {
                    uint32_t t[W / 2];
#pragma unroll
                    for (int w = 0; w < W; w += 2) {
                        const __nv_bfloat162 x = __floats2bfloat162_rn(v[w], v[w + 1]);
                        t[w / 2] = *reinterpret_cast<const uint32_t*>(&x);
                    }
                    store_words(smem + r * DH + col, t);
                    if (mine) store_words(cache + (size_t)pos * DH + col, t);
                };
                put(k0[e], newK, Kh, d);
                put(k1[e], newK, Kh, d + half);
                put(v0[e], newV, Vh, d);
                put(v1[e], newV, Vh, d + half);
            }
        }
    }

    float o[MT][2][4];
#pragma unroll
    for (int mt = 0; mt < MT; ++mt)
#pragma unroll
        for (int t = 0; t < 2; ++t)
#pragma unroll
            for (int e = 0; e < 4; ++e) o[mt][t][e] = 0.f;
    const int lrow = lane & 7, lmat = lane >> 3;          // ldmatrix: this lane addresses row lrow of matrix lmat
    const uint32_t qh_s = smem_u32(qh), ql_s = smem_u32(ql), ph_s = smem_u32(ph), pl_s = smem_u32(pl);

    // The q operand is the same for every tile: each warp keeps the A fragments of its row tile in
    // registers (high parts; the low parts too while a block is one row tile) instead of fetching
    // them from shared memory per tile, which is what bounded the score step.  A warp takes the row
    // tile mtw and MT groups of 8 keys of every tile.
    constexpr bool QLO_REG = MT == 1;
    const int mtw = MT == 1 ? 0 : warp >> 2;
    const int key0 = MT == 1 ? 8 * warp : 16 * (warp & 3);
    uint32_t qfh[DH / 16][4], qfl[QLO_REG ? DH / 16 : 1][4];
    __syncthreads();                        // the block's q rows are in shared memory
#pragma unroll
    for (int ks = 0; ks < DH / 16; ++ks) {
        const uint32_t aoff = (uint32_t)((mtw * 16 + (lmat & 1) * 8 + lrow) * C::QP + (2 * ks + (lmat >> 1)) * 16);
        ldsm_x4(qh_s + aoff, qfh[ks]);
        if (QLO_REG) ldsm_x4(ql_s + aoff, qfl[QLO_REG ? ks : 0]);
    }

    float run_m[R / 8], run_l[R / 8];       // running maximum and this lane's share of the running sum, rows warp + 8 i
#pragma unroll
    for (int i = 0; i < R / 8; ++i) { run_m[i] = -INFINITY; run_l[i] = 0.f; }
    bool failed = false;
    for (int it = 0; it < n_tiles; ++it) {
        const int st = it % STAGES, t0 = s_begin + it * TILE;
        const int ok = mbar_wait(&full[st], (uint32_t)(it / STAGES) & 1u);
        if (__syncthreads_or(!ok)) {
            if (!ok) mbar_wait(&full[st], (uint32_t)(it / STAGES) & 1u);
            failed = true;
            break;
        }
        // every thread is past the previous tile (the barrier above): its stage may be filled again
        if (tid == 0 && it >= 1 && it - 1 + STAGES < n_tiles) {
            fence_async_smem();
            request(it - 1 + STAGES);
        }
        unsigned char* Kt = Ks + st * C::TILE_BYTES;
        unsigned char* Vt = Vs + st * C::TILE_BYTES;
        const int valid = min(TILE, s_end - t0);
        const int new_lo = max(t0, n_old), n_new = t0 + valid - new_lo;
        if (n_new > 0 || valid < TILE) {       // same for every thread
            for (int idx = tid; idx < n_new * (DH / 8); idx += AT) {
                const int row = idx / (DH / 8), c = idx % (DH / 8), j = new_lo + row - t0, r = new_lo + row - n_old;
                *reinterpret_cast<uint4*>(Kt + kv_off<DH>(j, c)) = *reinterpret_cast<const uint4*>(newK + r * DH + c * 8);
                *reinterpret_cast<uint4*>(Vt + kv_off<DH>(j, c)) = *reinterpret_cast<const uint4*>(newV + r * DH + c * 8);
            }
            for (int idx = tid; idx < (TILE - valid) * (DH / 8); idx += AT) {
                const int j = valid + idx / (DH / 8), c = idx % (DH / 8);
                *reinterpret_cast<uint4*>(Vt + kv_off<DH>(j, c)) = make_uint4(0, 0, 0, 0);
            }
            __syncthreads();
        }
        // ---- scores of this warp's row tile against its MT groups of 8 keys; the high and low parts of q and
        //      the two halves of the head dimension accumulate separately, so that no chain is longer than DH/32 MMAs
        {
            float sacc2[MT][2][2][4];           // [key group][q part][half of the k steps]
#pragma unroll
            for (int g = 0; g < MT; ++g)
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    sacc2[g][0][0][e] = sacc2[g][0][1][e] = sacc2[g][1][0][e] = sacc2[g][1][1][e] = 0.f;
            const uint32_t Kt_s = smem_u32(Kt);
#pragma unroll
            for (int ks2 = 0; ks2 < DH / 32; ++ks2) {
#pragma unroll
                for (int g = 0; g < MT; ++g) {
                    uint32_t kb[4];
                    ldsm_x4(Kt_s + kv_off<DH>(key0 + 8 * g + lrow, 4 * ks2 + lmat), kb);
#pragma unroll
                    for (int hf = 0; hf < 2; ++hf) {
                        const int ks = 2 * ks2 + hf;
                        mma_bf16(sacc2[g][0][hf], qfh[ks], kb[2 * hf], kb[2 * hf + 1]);
                        if (QLO_REG) {
                            mma_bf16(sacc2[g][1][hf], qfl[QLO_REG ? ks : 0], kb[2 * hf], kb[2 * hf + 1]);
                        } else {
                            const uint32_t aoff = (uint32_t)((mtw * 16 + (lmat & 1) * 8 + lrow) * C::QP + (2 * ks + (lmat >> 1)) * 16);
                            uint32_t a[4];
                            ldsm_x4(ql_s + aoff, a);
                            mma_bf16(sacc2[g][1][hf], a, kb[2 * hf], kb[2 * hf + 1]);
                        }
                    }
                }
            }
#pragma unroll
            for (int g = 0; g < MT; ++g)
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const int r = mtw * 16 + (lane >> 2) + (e >> 1) * 8, j = key0 + 8 * g + (lane & 3) * 2 + (e & 1);
                    if (r < m) {
                        const int key = t0 + j, limit = p.causal ? n_keys + r : n_keys;
                        float s = -INFINITY;
                        bool vis = key < s_end && key < limit;
                        if (p.tree && key >= n_old) vis = key < s_end && ((p.tmask[r] >> (key - n_old)) & 1u);
                        if (vis) {
                            s = ((sacc2[g][1][0][e] + sacc2[g][1][1][e]) + (sacc2[g][0][0][e] + sacc2[g][0][1][e])) * p.scale;
                            if (bias_h) {
                                int bi = key - (sg.q_pos0 + r) + p.bias_zero;
                                bi = max(0, min(p.bias_len - 1, bi));
                                s += bias_h[bi];
                            }
                        }
                        sc[r * C::SP + j] = s;
                    }
                }
        }
        __syncthreads();
        // ---- online softmax: warp w owns rows w, w+8, ...; the weights leave as bf16 pairs.  The rows of a
        //      warp are independent, so their loads, shuffles and exponentials interleave; the row sums stay
        //      as per-lane partial sums until the walk is over.
        {
            float s0[R / 8], s1[R / 8], tmax[R / 8];
#pragma unroll
            for (int i = 0; i < R / 8; ++i) {
                const int r = warp + 8 * i;
                s0[i] = s1[i] = -INFINITY;
                if (r < m) { s0[i] = sc[r * C::SP + lane]; s1[i] = sc[r * C::SP + lane + 32]; }
                tmax[i] = fmaxf(s0[i], s1[i]);
            }
#pragma unroll
            for (int off = 16; off > 0; off >>= 1)
#pragma unroll
                for (int i = 0; i < R / 8; ++i) tmax[i] = fmaxf(tmax[i], __shfl_xor_sync(0xffffffffu, tmax[i], off));
#pragma unroll
            for (int i = 0; i < R / 8; ++i) {
                const int r = warp + 8 * i;
                if (r >= m) continue;
                const float old = run_m[i];
                const float nm = fmaxf(old, tmax[i]);
                float p0 = 0.f, p1 = 0.f, alpha = 1.f;
                if (nm > -INFINITY) {
                    p0 = expf(s0[i] - nm);
                    p1 = expf(s1[i] - nm);
                    alpha = expf(old - nm);
                }
                __nv_bfloat16 h0, l0, h1, l1;
                split2(p0, h0, l0);
                split2(p1, h1, l1);
                __nv_bfloat16* phr = reinterpret_cast<__nv_bfloat16*>(ph + r * C::PP);
                __nv_bfloat16* plr = reinterpret_cast<__nv_bfloat16*>(pl + r * C::PP);
                phr[lane] = h0; phr[lane + 32] = h1; plr[lane] = l0; plr[lane + 32] = l1;
                // the sum runs over the weights as the MMA will see them
                run_l[i] = run_l[i] * alpha + ((__bfloat162float(h0) + __bfloat162float(l0)) + (__bfloat162float(h1) + __bfloat162float(l1)));
                run_m[i] = nm;
                if (lane == 0) row_a[r] = alpha;
            }
        }
        __syncthreads();
        // ---- P.V for output dimensions 16*warp .. 16*warp+15
        if (warp < DH / 16) {
#pragma unroll
            for (int mt = 0; mt < MT; ++mt) {
                const float a0 = row_a[mt * 16 + (lane >> 2)], a1 = row_a[mt * 16 + (lane >> 2) + 8];
#pragma unroll
                for (int t = 0; t < 2; ++t) { o[mt][t][0] *= a0; o[mt][t][1] *= a0; o[mt][t][2] *= a1; o[mt][t][3] *= a1; }
            }
            const uint32_t Vt_s = smem_u32(Vt);
            float ol[MT][2][4];                 // the low parts of the weights accumulate on their own chain
#pragma unroll
            for (int mt = 0; mt < MT; ++mt)
#pragma unroll
                for (int t = 0; t < 2; ++t)
#pragma unroll
                    for (int e = 0; e < 4; ++e) ol[mt][t][e] = 0.f;
#pragma unroll
            for (int ks = 0; ks < TILE / 16; ++ks) {
                uint32_t vb[4];
                ldsm_x4_t(Vt_s + kv_off<DH>(16 * ks + (lmat & 1) * 8 + lrow, 2 * warp + (lmat >> 1)), vb);
#pragma unroll
                for (int mt = 0; mt < MT; ++mt) {
                    const uint32_t aoff = (uint32_t)((mt * 16 + (lmat & 1) * 8 + lrow) * C::PP + (2 * ks + (lmat >> 1)) * 16);
                    uint32_t a[4];
                    ldsm_x4(ph_s + aoff, a);
                    mma_bf16(o[mt][0], a, vb[0], vb[1]);
                    mma_bf16(o[mt][1], a, vb[2], vb[3]);
                    ldsm_x4(pl_s + aoff, a);
                    mma_bf16(ol[mt][0], a, vb[0], vb[1]);
                    mma_bf16(ol[mt][1], a, vb[2], vb[3]);
                }
            }
#pragma unroll
            for (int mt = 0; mt < MT; ++mt)
#pragma unroll
                for (int t = 0; t < 2; ++t)
#pragma unroll
                    for (int e = 0; e < 4; ++e) o[mt][t][e] += ol[mt][t][e];
        }
    }
    if (failed && tid == 0) set_status(p.status, CSD_ERR_TIMEOUT);
#pragma unroll
    for (int i = 0; i < R / 8; ++i) {
        const float l = warp_sum(run_l[i]);
        const int r = warp + 8 * i;
        if (lane == 0 && r < m) { row_m[r] = run_m[i]; row_l[r] = l; }
    }
    __syncthreads();


    // element (mt, t, e) of `o`: row mt*16 + lane/4 (+8 for e >= 2), dimension 16*warp + 8*t + 2*(lane%4) + (e&1)
    if (p.nsplit == 1) {
        if (warp < DH / 16) {
#pragma unroll
            for (int mt = 0; mt < MT; ++mt)
#pragma unroll
                for (int hr = 0; hr < 2; ++hr) {
                    const int r = mt * 16 + (lane >> 2) + hr * 8;
                    if (r >= m) continue;
                    const float inv = row_l[r] > 0.f ? 1.f / row_l[r] : 0.f;
#pragma unroll
                    for (int t = 0; t < 2; ++t) {
                        const int d = 16 * warp + 8 * t + 2 * (lane & 3);
                        const float a = o[mt][t][2 * hr] * inv, b = o[mt][t][2 * hr + 1] * inv;
                        if (p.out_xs) store_split(p.out_xs, p.out_xs_ld, p.xs_m, sg.xs_r0 + r, h * DH + d, a, b);
                        else *reinterpret_cast<float2*>(sg.out + (size_t)r * p.ldo + h * DH + d) = make_float2(a, b);
                    }
                }
        }
        return;
    }
    float* rec = reinterpret_cast<float*>(qh);      // q is not needed any more (all threads are past the last tile)
    if (warp < DH / 16) {
#pragma unroll
        for (int mt = 0; mt < MT; ++mt)
#pragma unroll
            for (int hr = 0; hr < 2; ++hr) {
                const int r = mt * 16 + (lane >> 2) + hr * 8;
                if (r >= m) continue;
#pragma unroll
                for (int t = 0; t < 2; ++t) {
                    const int d = 16 * warp + 8 * t + 2 * (lane & 3);
                    *reinterpret_cast<float2*>(rec + r * C::REC + d) = make_float2(o[mt][t][2 * hr], o[mt][t][2 * hr + 1]);
                }
            }
    }
    if (tid < m) { rec[tid * C::REC + DH] = row_m[tid]; rec[tid * C::REC + DH + 1] = row_l[tid]; }
    cluster.sync();
    merge_splits<DH, C::REC>(cluster, rec, p, sg.out, sg.xs_r0, h, split, m);
    cluster.sync();       // no CTA leaves while another may still read its record
}
static bool g_attn_cuda_cores = false;
void set_attention_cuda_cores(bool on) { g_attn_cuda_cores = on; }
bool row_attention_supported(int Dh) { return (Dh == 64 || Dh == 128) && !g_attn_cuda_cores; }

// Splits per head: one 64-key tile per CTA while that keeps the splits of a head inside one portable cluster (8) and the
// grid near two CTAs per SM (short caches are latency-bound, and more splits mean more tiles in flight at once); long
// caches walk several tiles per CTA, two requests ahead.  At head dimension 128 (8 layers of the 7B shape, 32 heads, us):
//   up to 5 rows, caches of 5 to 8 tiles do with about a CTA per SM, each walking two (300 keys: 704 with 3 splits, 709 with 5;
//     400: 709 with 4, 714 with 7); on longer ones 7 and 8 splits are level (1000 keys 742 both, 1500 757 and 763).  At 6 to 8 rows
//     the half is level too, larger blocks want the splits (9 rows, 300 keys: 772 with 3, 757 with 5).
//   from 6 rows on, at most 7: 6 rows 1000 keys 752 with 7, 782 with 8; 8 rows 769 and 800, 1500 keys 785 and 824; 17 rows 1000 keys
//     918 and 974, 1500 keys 949 and 1022.  (At 2048 keys 8 splits of whole tiles are 7 anyway.)
int attn_splits(int total_keys, int H, int Dh, int gemm_rows) {
    const int sms = tc_sm_count(), by_sm = (2 * sms + H - 1) / H, tiles = (total_keys + TILE - 1) / TILE;
    int n = by_sm < tiles ? by_sm : tiles;
    if (n > MAX_SPLITS) n = MAX_SPLITS;
    if (Dh == 128 && gemm_rows > 5 && n == MAX_SPLITS) n = MAX_SPLITS - 1;
    if (Dh == 128 && gemm_rows <= 5 && n == tiles && tiles > 4 && H * tiles > sms) n = (tiles + 1) / 2;
    return n < 1 ? 1 : n;
}

static void attn_launch_config(cudaLaunchConfig_t& cfg, cudaLaunchAttribute* attr, const AttnParams& ap, size_t smem,
                               cudaStream_t st) {
    cfg = cudaLaunchConfig_t{};
    cfg.gridDim = dim3((unsigned)ap.H, (unsigned)ap.nsplit);
    cfg.blockDim = dim3(AT);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;      // the splits of one head exchange results on chip
    attr[1].val.clusterDim.x = 1; attr[1].val.clusterDim.y = (unsigned)ap.nsplit; attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
}

template <int DH>
static csd_status launch_dh(const AttnParams& ap, cudaStream_t st) {
    auto kern = block_attention_kernel<DH>;
    static PerDevice ready;
    const csd_status ok = allow_smem(ready, kern, AttnCfg<DH>::SMEM);
    if (ok != CSD_OK) return ok;
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr[2];
    attn_launch_config(cfg, attr, ap, AttnCfg<DH>::SMEM, st);
    CSD_CUDA(cudaLaunchKernelEx(&cfg, kern, ap));
    count_launch();
    return CSD_OK;
}

template <int DH, int MT>
static csd_status launch_mma(const AttnSegs& segs, int nseg, const AttnParams& ap, cudaStream_t st) {
    auto kern = block_attention_mma_kernel<DH, MT>;
    static PerDevice ready;
    const size_t smem = MmaCfg<DH>::smem(MT * 16);
    const csd_status ok = allow_smem(ready, kern, smem);
    if (ok != CSD_OK) return ok;
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr[2];
    attn_launch_config(cfg, attr, ap, smem, st);
    cfg.gridDim.z = (unsigned)nseg;
    CSD_CUDA(cudaLaunchKernelEx(&cfg, kern, segs, ap));
    count_launch();
    return CSD_OK;
}

static csd_status launch_attention_block(const AttnArgs* a, int n, cudaStream_t st);

// Blocks of more than MAXM rows over a cache that already holds their keys (wide passes whose head dimension has no
// launch_row_attention): one launch per MAXM rows.
csd_status launch_attention(const AttnArgs& a, cudaStream_t st) {
    if (a.m <= MAXM) return launch_attention_block(&a, 1, st);
    if (a.k_new || a.tree_mask || a.out_xs || a.m > CSD_WIDE_ROWS) return CSD_ERR_INVALID_ARG;
    for (int r0 = 0; r0 < a.m; r0 += MAXM) {
        AttnArgs s = a;
        s.q = a.q + (size_t)r0 * a.ldq; s.m = a.m - r0 < MAXM ? a.m - r0 : MAXM;
        s.n_keys = a.causal ? a.n_keys + r0 : a.n_keys;
        s.q_pos0 = a.q_pos0 + r0;
        s.out = a.out + (size_t)r0 * a.ldo;
        const csd_status rc = launch_attention_block(&s, 1, st);
        if (rc != CSD_OK) return rc;
    }
    return CSD_OK;
}

csd_status launch_attention_batch(const AttnArgs* a, int n, int* taken, cudaStream_t st) {
    int cnt = n > 1 && (a[0].Dh == 64 || a[0].Dh == 128) && !g_attn_cuda_cores ? (n < MAX_SEGS ? n : MAX_SEGS) : 1;
    for (int j = 0; j < cnt; ++j)
        if (a[j].tree_mask || a[j].m > 16) cnt = 1;
    *taken = cnt;
    return cnt == 1 ? launch_attention(a[0], st) : launch_attention_block(a, cnt, st);
}

// The blocks of n sequences of one model (n <= MAX_SEGS; more than one on the tensor-core kernel only, without a tree).
static csd_status launch_attention_block(const AttnArgs* args, int n, cudaStream_t st) {
    const AttnArgs& a = args[0];
    int longest = 0, rows = 0, totals[MAX_SEGS];
    for (int i = 0; i < n; ++i) {
        const AttnArgs& b = args[i];
        if (!b.q || !b.Kc || !b.Vc || !b.out || b.m < 1 || b.m > MAXM || b.H < 1 || b.n_keys < 0) return CSD_ERR_INVALID_ARG;
        const bool append = b.k_new != nullptr;
        if (append && (!b.v_new || !b.causal || b.n_keys < 1)) return CSD_ERR_INVALID_ARG;
        if ((b.rope_cos != nullptr) != (b.rope_sin != nullptr) || (b.rope_cos && !append)) return CSD_ERR_INVALID_ARG;
        if ((((uintptr_t)b.Kc) & 15) || (((uintptr_t)b.Vc) & 15)) return CSD_ERR_INVALID_ARG;
        // (rows are read and written four values at a time)
        if ((((uintptr_t)b.q) & 15) || (((uintptr_t)b.k_new) & 15) || (((uintptr_t)b.v_new) & 15) || (((uintptr_t)b.out) & 15) || (((uintptr_t)b.out_xs) & 15) ||
            (b.ldq & 3) || (b.ld_new & 3) || (b.ldo & 3) || (b.out_xs_ld & 3))
            return CSD_ERR_INVALID_ARG;
        totals[i] = b.causal ? b.n_keys + b.m - 1 : b.n_keys;
        if (totals[i] < 1 || totals[i] > b.cap) return CSD_ERR_CAPACITY;
        if (totals[i] > longest) longest = totals[i];
        if (b.m > rows) rows = b.m;
    }
    const bool append = a.k_new != nullptr;
    AttnParams ap;
    ap.q = a.q; ap.k_new = a.k_new; ap.v_new = a.v_new; ap.ld_new = a.ld_new; ap.rope_cos = a.rope_cos;
    ap.rope_sin = a.rope_sin; ap.Kc = a.Kc; ap.Vc = a.Vc; ap.bias = a.bias; ap.out = a.out;
    ap.status = status_word_device();
    ap.ldq = a.ldq; ap.m = a.m; ap.cap = a.cap; ap.H = a.H; ap.n_keys = a.n_keys;
    ap.n_old = append ? a.n_keys - 1 : totals[0];
    ap.early_loads = a.kv_settled ? 1 : 0;
    ap.causal = a.causal; ap.bias_len = a.bias_len; ap.bias_zero = a.bias_zero; ap.q_pos0 = a.q_pos0;
    ap.ldo = a.ldo; ap.scale = a.scale; ap.out_xs = a.out_xs; ap.out_xs_ld = a.out_xs_ld;
    ap.xs_m = a.out_xs_rows > 0 ? a.out_xs_rows : a.m; ap.xs_r0 = a.out_xs_row0;
    ap.tree = 0;
    if (a.tree_mask) {
        if (!append || !a.tree_depth || a.bias) return CSD_ERR_INVALID_ARG;
        ap.tree = 1;
        for (int r = 0; r < MAXM; ++r) { ap.tmask[r] = r < a.m ? a.tree_mask[r] : 0u; ap.tdepth[r] = r < a.m ? (unsigned char)a.tree_depth[r] : 0; }
    }
    // every sequence's splits share one cluster shape, set by the longest cache; shorter ones leave their last splits empty
    ap.nsplit = attn_splits(longest, a.H * n, a.Dh, a.out_xs_rows > 0 ? a.out_xs_rows : a.m);
    auto split_len = [&](int total) { return ((total + ap.nsplit - 1) / ap.nsplit + TILE - 1) / TILE * TILE; };
    ap.nsplit = (longest + split_len(longest) - 1) / split_len(longest);
    ap.split_len = split_len(totals[0]);
    // head dimensions 64 and 128 run on the tensor cores; the caches then need tensor maps (rows = all heads' positions)
    if ((a.Dh == 64 || a.Dh == 128) && !g_attn_cuda_cores) {
        AttnSegs segs;
        bool maps = true;
        for (int i = 0; i < n; ++i) {
            const AttnArgs& b = args[i];
            maps = maps && tensor_map_2d(b.Kc, b.H * b.cap, b.Dh, TILE, &segs.k[i]) && tensor_map_2d(b.Vc, b.H * b.cap, b.Dh, TILE, &segs.v[i]);
            segs.seg[i] = AttnSeg{b.q, b.k_new, b.v_new, b.Kc, b.Vc, b.out, b.m, b.n_keys, b.k_new ? b.n_keys - 1 : totals[i],
                                  split_len(totals[i]), b.q_pos0, b.out_xs_row0};
        }
        if (maps) {
            if (a.Dh == 64) return rows <= 16 ? launch_mma<64, 1>(segs, n, ap, st) : launch_mma<64, 2>(segs, n, ap, st);
            return rows <= 16 ? launch_mma<128, 1>(segs, n, ap, st) : launch_mma<128, 2>(segs, n, ap, st);
        }
    }
    if (n > 1) return CSD_ERR_UNSUPPORTED;
    switch (a.Dh) {
        case 32: return launch_dh<32>(ap, st);
        case 64: return launch_dh<64>(ap, st);
        case 128: return launch_dh<128>(ap, st);
    }
    return CSD_ERR_SHAPE;
}

}  // namespace csd

extern "C" csd_status csd_set_attention_path(int path) {
    if (path < 0 || path > 1) return CSD_ERR_INVALID_ARG;
    csd::set_attention_cuda_cores(path == 1);
    return CSD_OK;
}
