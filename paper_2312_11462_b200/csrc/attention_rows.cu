// Attention of the many rows of a prompt or source pass against a bf16 K/V cache that already holds their keys.
//
// grid = (heads, blocks of 64 rows), the blocks that see most keys first; four warps of 16 rows each.  K and V come
// in 64-key tiles by tensor-map TMA (three stages, one thread requests, warps hand stages back on an mbarrier), so
// nothing in the walk is block-wide: a warp keeps its rows' q fragments, online softmax and output in registers,
// and the accumulator fragments of q.K^T are the operand fragments of P.V.  q (rotated here, from its fp32
// projection) and the softmax weights are bf16 pairs, two MMAs each.  The output leaves through shared
// memory in whole 16-byte pieces, as the two-term rows of the projection that follows.
//
// What bounds it: the MMAs (256 per warp and tile) and the softmax's instructions between them, two CTAs an SM
// taking turns.  1000 rows on an empty cache, 32 heads of 128: 72 us (230 TFLOP/s of two-term products), against 228 us
// for the same walk in blocks of 32 rows whose scores and weights crossed shared memory under three block barriers a tile.
#include "attention.cuh"
#include "attention_mma.cuh"
#include "gemm_tc.cuh"

namespace csd {

constexpr int RW = 4, RROWS = 16 * RW;      // warps and rows of a CTA
constexpr int RSTAGES = 3;

struct RowsParams {
    const float* q; const float* rope_cos; const float* rope_sin; const float* bias;
    __nv_bfloat16* xs; int* status;
    int ldq, m, cap, n_keys, causal, bias_len, bias_zero, q_pos0, xs_ld, xs_rows;
    float scale;
};

template <int DH> struct RowsCfg {
    static constexpr size_t TILE_BYTES = (size_t)TILE * DH * 2;
    static constexpr size_t SMEM = 1024 + 2 * RSTAGES * TILE_BYTES + 2 * RSTAGES * 8;
    static constexpr int OP = DH * 4 + 16;                 // bytes of an output row: two terms, one 16-byte skew
    static_assert(RROWS * OP <= 2 * RSTAGES * (int)TILE_BYTES, "the output rows fit the stages");
};

template <int DH>
__global__ void __launch_bounds__(32 * RW, 2)
row_attention_kernel(const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmV, const RowsParams p) {
    using C = RowsCfg<DH>;
    constexpr int KS = DH / 16, NB = DH / 64, HALF = DH / 2;
    extern __shared__ unsigned char smem_dyn[];
    unsigned char* base = (unsigned char*)(((uintptr_t)smem_dyn + 1023) & ~(uintptr_t)1023);
    unsigned char* Vs = base + RSTAGES * C::TILE_BYTES;
    uint64_t* full = reinterpret_cast<uint64_t*>(Vs + RSTAGES * C::TILE_BYTES);
    uint64_t* empty = full + RSTAGES;

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int h = blockIdx.x, blk = (int)gridDim.y - 1 - (int)blockIdx.y;
    const int r0 = blk * RROWS, rows = min(RROWS, p.m - r0);
    const int total = p.causal ? p.n_keys + r0 + rows - 1 : p.n_keys;       // keys the block's last row sees
    const int n_tiles = (total + TILE - 1) / TILE;

    if (tid == 0) {
        for (int s = 0; s < RSTAGES; ++s) { mbar_init(&full[s], 1); mbar_init(&empty[s], RW); }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    pdl_wait();
    pdl_trigger();

    auto request = [&](int it) {
        const int st = it % RSTAGES, row = h * p.cap + it * TILE;
        mbar_expect_tx(&full[st], 2 * (uint32_t)C::TILE_BYTES);
#pragma unroll
        for (int b = 0; b < NB; ++b) tma_load_2d(base + st * C::TILE_BYTES + b * (TILE * 128), &tmK, &full[st], b * 64, row);
#pragma unroll
        for (int b = 0; b < NB; ++b) tma_load_2d(Vs + st * C::TILE_BYTES + b * (TILE * 128), &tmV, &full[st], b * 64, row);
    };
    if (tid == 0)
        for (int it = 0; it < RSTAGES - 1 && it < n_tiles; ++it) request(it);

    // ---- q fragments: this lane holds rows ra and ra + 8 of the block, dimensions 16 ks + 2 (lane % 4) + {0, 1, 8, 9}; the
    //      partner of a dimension under the rotation is HALF further on, in fragment ks + KS / 2 of the same lane
    const int ra = warp * 16 + (lane >> 2), c0 = 2 * (lane & 3);
    uint32_t qh[KS][4], ql[KS][4];
#pragma unroll
    for (int hr = 0; hr < 2; ++hr) {
        const int r = min(r0 + ra + 8 * hr, p.m - 1);                        // (rows past the last repeat it; nothing of them is stored)
        const float* src = p.q + (size_t)r * p.ldq + h * DH;
#pragma unroll
        for (int ks = 0; ks < KS / 2; ++ks)
#pragma unroll
            for (int cc = 0; cc < 2; ++cc) {
                const int d = 16 * ks + 8 * cc + c0;
                float2 a = *reinterpret_cast<const float2*>(src + d), b = *reinterpret_cast<const float2*>(src + d + HALF);
                if (p.rope_cos) {
                    const size_t at = (size_t)(p.q_pos0 + r) * HALF + d;
                    const float2 c = *reinterpret_cast<const float2*>(p.rope_cos + at), s = *reinterpret_cast<const float2*>(p.rope_sin + at);
                    const float2 x = a, y = b;
                    a = make_float2(x.x * c.x - y.x * s.x, x.y * c.y - y.y * s.y);
                    b = make_float2(x.x * s.x + y.x * c.x, x.y * s.y + y.y * c.y);
                }
                pack_pair(a.x, a.y, qh[ks][2 * cc + hr], ql[ks][2 * cc + hr]);
                pack_pair(b.x, b.y, qh[ks + KS / 2][2 * cc + hr], ql[ks + KS / 2][2 * cc + hr]);
            }
    }

    float o[2 * KS][4];
#pragma unroll
    for (int t = 0; t < 2 * KS; ++t) o[t][0] = o[t][1] = o[t][2] = o[t][3] = 0.f;
    float run_m[2] = {-INFINITY, -INFINITY}, run_l[2] = {0.f, 0.f};          // running maximum, this lane's share of the running sum
    const int lrow = lane & 7, lmat = lane >> 3;                             // ldmatrix: this lane addresses row lrow of matrix lmat
    // A tile's biases depend on key - row only: the warp's 79 values of a tile, lanes' loads in flight during the score MMAs
    __shared__ float bias_w[RW][96];
    const float* bias_h = p.bias ? p.bias + (size_t)h * p.bias_len : nullptr;
    const int bias0 = p.bias_zero - (p.q_pos0 + r0 + warp * 16 + 15);        // table index of key 0 for the warp's last row
    const int lim_lo = p.causal ? p.n_keys + r0 + warp * 16 : p.n_keys;      // keys the warp's first row sees, and its last
    const int lim_hi = warp * 16 >= rows ? 0 : (p.causal ? min(lim_lo + 15, total) : p.n_keys);
    bool failed = false;

#pragma unroll 1
    for (int it = 0; it < n_tiles; ++it) {
        const int st = it % RSTAGES, t0 = it * TILE, next = it + RSTAGES - 1;
        bool ok = true;
        if (tid == 0 && next < n_tiles) {
            ok = next < RSTAGES || mbar_wait(&empty[next % RSTAGES], (uint32_t)(next / RSTAGES - 1) & 1u);
            if (ok) request(next);
        }
        ok = ok && mbar_wait(&full[st], (uint32_t)(it / RSTAGES) & 1u);
        if (__any_sync(0xffffffffu, !ok)) { failed = true; break; }
        const uint32_t Kt = smem_u32(base + st * C::TILE_BYTES), Vt = smem_u32(Vs + st * C::TILE_BYTES);
        if (total - t0 < TILE) {              // last tile: what lies behind the block's keys may be anything, also not a number
            const int valid = total - t0;
            for (int i = tid; i < (TILE - valid) * (DH / 8); i += 32 * RW)
                *reinterpret_cast<uint4*>(Vs + st * C::TILE_BYTES + kv_off<DH>(valid + i / (DH / 8), i % (DH / 8))) = make_uint4(0, 0, 0, 0);
            __syncthreads();
        }
        if (t0 < lim_hi) {
            float bw[3];
            if (bias_h)
#pragma unroll
                for (int i = 0; i < 3; ++i) bw[i] = bias_h[max(0, min(p.bias_len - 1, bias0 + t0 + 32 * i + lane))];
            // ---- scores: four key groups at a time, so that an accumulator's next MMA is four MMAs away
            float s[8][4];
#pragma unroll
            for (int g = 0; g < 8; ++g) s[g][0] = s[g][1] = s[g][2] = s[g][3] = 0.f;
#pragma unroll
            for (int k2 = 0; k2 < KS / 2; ++k2)
#pragma unroll
                for (int g4 = 0; g4 < 8; g4 += 4) {
                    uint32_t kb[4][4];
#pragma unroll
                    for (int g = 0; g < 4; ++g) ldsm_x4(Kt + kv_off<DH>(8 * (g4 + g) + lrow, 4 * k2 + lmat), kb[g]);
#pragma unroll
                    for (int hf = 0; hf < 2; ++hf) {
#pragma unroll
                        for (int g = 0; g < 4; ++g) mma_bf16(s[g4 + g], ql[2 * k2 + hf], kb[g][2 * hf], kb[g][2 * hf + 1]);
#pragma unroll
                        for (int g = 0; g < 4; ++g) mma_bf16(s[g4 + g], qh[2 * k2 + hf], kb[g][2 * hf], kb[g][2 * hf + 1]);
                    }
                }
            if (bias_h) {
                __syncwarp();
#pragma unroll
                for (int i = 0; i < 3; ++i) bias_w[warp][32 * i + lane] = bw[i];
                __syncwarp();
            }
            // ---- scale, bias, mask
            const bool edge = t0 + TILE > (p.causal ? lim_lo : total);       // some row of the warp does not see the whole tile
#pragma unroll
            for (int g = 0; g < 8; ++g)
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    s[g][e] *= p.scale;
                    if (bias_h || edge) {
                        const int j = 8 * g + c0 + (e & 1), rr = (lane >> 2) + 8 * (e >> 1), key = t0 + j, r = r0 + warp * 16 + rr;
                        if (bias_h) s[g][e] += bias_w[warp][j + 15 - rr];
                        if (key >= total || (p.causal && key >= p.n_keys + r)) s[g][e] = -INFINITY;
                    }
                }
            // ---- online softmax of the lane's two rows (every row sees key 0, so the maximum is finite)
#pragma unroll
            for (int hr = 0; hr < 2; ++hr) {
                float mx = s[0][2 * hr];
#pragma unroll
                for (int g = 0; g < 8; ++g) mx = fmaxf(mx, fmaxf(s[g][2 * hr], s[g][2 * hr + 1]));
                mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
                mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
                const float nm = fmaxf(run_m[hr], mx);
                const float alpha = expf(run_m[hr] - nm);
                run_m[hr] = nm;
                run_l[hr] *= alpha;
#pragma unroll
                for (int g = 0; g < 8; ++g) {
                    s[g][2 * hr] = expf(s[g][2 * hr] - nm);
                    s[g][2 * hr + 1] = expf(s[g][2 * hr + 1] - nm);
                }
#pragma unroll
                for (int t = 0; t < 2 * KS; ++t) { o[t][2 * hr] *= alpha; o[t][2 * hr + 1] *= alpha; }
            }
            // ---- P.V, 16 keys at a time; the row sums run over the weights as the MMAs see them
#pragma unroll
            for (int kk = 0; kk < TILE / 16; ++kk) {
                uint32_t ph[4], pl[4];
#pragma unroll
                for (int f = 0; f < 4; ++f) {
                    const float x = s[2 * kk + (f >> 1)][2 * (f & 1)], y = s[2 * kk + (f >> 1)][2 * (f & 1) + 1];
                    pack_pair(x, y, ph[f], pl[f]);
                    run_l[f & 1] += (bf16lo(ph[f]) + bf16lo(pl[f])) + (bf16hi(ph[f]) + bf16hi(pl[f]));
                }
#pragma unroll
                for (int d2 = 0; d2 < KS; d2 += 2) {
                    uint32_t vb[2][4];
#pragma unroll
                    for (int u = 0; u < 2; ++u) ldsm_x4_t(Vt + kv_off<DH>(16 * kk + (lmat & 1) * 8 + lrow, 2 * (d2 + u) + (lmat >> 1)), vb[u]);
#pragma unroll
                    for (int u = 0; u < 4; ++u) mma_bf16(o[2 * d2 + u], pl, vb[u >> 1][2 * (u & 1)], vb[u >> 1][2 * (u & 1) + 1]);
#pragma unroll
                    for (int u = 0; u < 4; ++u) mma_bf16(o[2 * d2 + u], ph, vb[u >> 1][2 * (u & 1)], vb[u >> 1][2 * (u & 1) + 1]);
                }
            }
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(&empty[st]);
    }
    if (failed) {
        set_status(p.status, CSD_ERR_TIMEOUT);
        __nanosleep(2000000);              // let copies already in flight land before the CTA's memory is released
    }
    __syncthreads();                       // every tile has been read: the stages take the output rows
    unsigned char* orow = base;
#pragma unroll
    for (int hr = 0; hr < 2; ++hr) {
        float l = run_l[hr];
        l += __shfl_xor_sync(0xffffffffu, l, 1);
        l += __shfl_xor_sync(0xffffffffu, l, 2);
        const float inv = l > 0.f ? 1.f / l : 0.f;
        unsigned char* dst = orow + (size_t)(ra + 8 * hr) * C::OP;
#pragma unroll
        for (int t = 0; t < 2 * KS; ++t) {
            const float x = o[t][2 * hr] * inv, y = o[t][2 * hr + 1] * inv;
            uint32_t w1, w2;
            pack_pair(x, y, w1, w2);
            *reinterpret_cast<uint32_t*>(dst + (8 * t + c0) * 2) = w1;
            *reinterpret_cast<uint32_t*>(dst + DH * 2 + (8 * t + c0) * 2) = w2;
        }
    }
    __syncwarp();                          // a warp stores its own rows
    constexpr int PER = DH / 4;            // 16-byte pieces of an output row
    for (int i = lane; i < 16 * PER; i += 32) {
        const int r = warp * 16 + i / PER, c = i % PER;
        if (r >= rows) break;
        const uint4 v = *reinterpret_cast<const uint4*>(orow + (size_t)r * C::OP + c * 16);
        const int term = c / (PER / 2), cc = c % (PER / 2);
        *reinterpret_cast<uint4*>(p.xs + ((size_t)term * p.xs_rows + r0 + r) * p.xs_ld + h * DH + cc * 8) = v;
    }
}

template <int DH>
static csd_status launch_rows(const CUtensorMap& tk, const CUtensorMap& tv, const RowsParams& rp, int H, cudaStream_t st) {
    auto kern = row_attention_kernel<DH>;
    static PerDevice ready;
    const csd_status ok = allow_smem(ready, kern, RowsCfg<DH>::SMEM);
    if (ok != CSD_OK) return ok;
    PdlLaunch L(dim3((unsigned)H, (unsigned)((rp.m + RROWS - 1) / RROWS)), dim3(32 * RW), RowsCfg<DH>::SMEM, st);
    CSD_CUDA(cudaLaunchKernelEx(&L.cfg, kern, tk, tv, rp));
    count_launch();
    return CSD_OK;
}

csd_status launch_row_attention(const AttnArgs& a, cudaStream_t st) {
    if (!a.q || !a.Kc || !a.Vc || !a.out_xs2 || a.m < 1 || a.m > CSD_WIDE_ROWS || a.H < 1 || a.n_keys < 1 || (a.Dh != 64 && a.Dh != 128))
        return CSD_ERR_INVALID_ARG;
    if ((a.ldq & 1) || (((uintptr_t)a.q) & 7) || (((uintptr_t)a.Kc) & 15) || (((uintptr_t)a.Vc) & 15)) return CSD_ERR_INVALID_ARG;
    if ((a.out_xs_ld & 7) || (((uintptr_t)a.out_xs2) & 15)) return CSD_ERR_INVALID_ARG;
    if ((a.causal ? a.n_keys + a.m - 1 : a.n_keys) > a.cap) return CSD_ERR_CAPACITY;
    CUtensorMap tk, tv;
    if (!tensor_map_2d(a.Kc, a.H * a.cap, a.Dh, TILE, &tk) || !tensor_map_2d(a.Vc, a.H * a.cap, a.Dh, TILE, &tv)) return CSD_ERR_UNSUPPORTED;
    RowsParams rp;
    rp.q = a.q; rp.rope_cos = a.q_rope_cos; rp.rope_sin = a.q_rope_sin; rp.bias = a.bias; rp.xs = a.out_xs2;
    rp.status = status_word_device();
    rp.ldq = a.ldq; rp.m = a.m; rp.cap = a.cap; rp.n_keys = a.n_keys; rp.causal = a.causal; rp.bias_len = a.bias_len;
    rp.bias_zero = a.bias_zero; rp.q_pos0 = a.q_pos0; rp.xs_ld = a.out_xs_ld; rp.xs_rows = a.out_xs_rows;
    rp.scale = a.scale;
    return a.Dh == 64 ? launch_rows<64>(tk, tv, rp, a.H, st) : launch_rows<128>(tk, tv, rp, a.H, st);
}

}  // namespace csd
