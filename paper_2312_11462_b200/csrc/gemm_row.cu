// Row variant of the weight-streaming GEMM  Y[m, N] = X[m, K] . W[N, K]^T  for the matrices of draft
// models (K <= 3072): whole weight rows per warp, fp32 FMA, nothing shared between CTAs.
//
// Such a GEMM is bound by the chain of dependent steps, not by bytes (2304 x 768: 3.5 MB, 0.6 us at the copy
// rate): launch, wait for the kernel that produces the rows, fetch the rows, multiply, reduce, store.  The
// kernel keeps that chain short.  A warp requests its R weight rows over all of K into registers before the
// dependency wait; after it the CTA fetches the block's rows (all loads of a warp at once) into shared
// memory, times the gain of the RMS norm, with the sums of squares taken on the way; the R x m sums are reduced over the
// lanes by a butterfly that leaves sum v in lane v, which finishes it.  One barrier in all, no partial sums.
// Measured (back to back, 1 row): 2304 x 768 1.9 us, 768 x 3072 2.4 us, 32000 x 768 (49 MB) 8.4 us = 5.9 TB/s; the
// tensor-core kernel 7.4, 7.6 and 14.2 us.  Packed fp32 FMAs gave nothing, cp.async staging cost 1 us a launch.
#include "gemm_tc.cuh"

namespace csd {

constexpr int RW_THREADS = 256, RW_WARPS = RW_THREADS / 32;
constexpr int RW_STEP = 256;               // K elements a warp covers per 16-byte load
constexpr int RW_MAX_STEPS = 12;
constexpr size_t RW_SMEM_MAX = 110 * 1024; // two CTAs share an SM

struct RowParams {
    const __nv_bfloat16* W; const __nv_bfloat16* W2; const float* X; const __nv_bfloat16* gain; float* Y;
    const int32_t* tokens; const __nv_bfloat16* embed; float* x_out; int* status; unsigned* tickets;
    int N, K, ldx, ldy, m, steps, epilogue, vocab, n_clear;
    float eps;
};

static int row_m(int m) { return m <= 6 ? m : 8; }
static size_t row_smem(int M, int steps) { return (size_t)M * steps * RW_STEP * sizeof(float) + (size_t)steps * RW_STEP * 2 + (size_t)M * RW_MAX_STEPS * sizeof(float); }

// Shapes the kernel takes: all of K in a warp's registers, the rows in shared memory.
bool row_supported(int m, int N, int K, bool dual) {
    if (m < 1 || m > 8 || N < 1 || K < 8 || (K & 7)) return false;
    const int steps = (K + RW_STEP - 1) / RW_STEP;
    return steps <= (dual ? 3 : RW_MAX_STEPS) && row_smem(row_m(m), steps) <= RW_SMEM_MAX;
}

// sums over the lanes of V <= 32 values each; lane v returns the sum of value v (garbage beyond V)
template <int V>
__device__ __forceinline__ float lane_sums(float (&v)[V], int lane) {
    constexpr int P = V <= 1 ? 1 : V <= 2 ? 2 : V <= 4 ? 4 : V <= 8 ? 8 : V <= 16 ? 16 : 32;
    float a[P];
#pragma unroll
    for (int i = 0; i < P; ++i) a[i] = i < V ? v[i < V ? i : 0] : 0.f;
#pragma unroll
    for (int n = P / 2; n >= 1; n >>= 1)             // lanes whose bit n is set keep the upper half of the values
#pragma unroll
        for (int i = 0; i < n; ++i) {
            const bool up = (lane & n) != 0;
            const float give = up ? a[i] : a[i + n], keep = up ? a[i + n] : a[i];
            a[i] = keep + __shfl_xor_sync(0xffffffffu, give, n);
        }
#pragma unroll
    for (int o = P; o < 32; o <<= 1) a[0] += __shfl_xor_sync(0xffffffffu, a[0], o);
    return a[0];
}

// M: rows of X (m rounded up, the rest zero), R: weight rows a warp takes at a time, S: most K steps; GATHER: the rows are
// those of the embedding table that the tokens name
template <int M, int R, int S, bool DUAL, bool GATHER>
__global__ void __launch_bounds__(RW_THREADS, 2)
row_gemm_kernel(const RowParams p) {
    constexpr int NT = DUAL ? 2 : 1, V = R * M, Q = (V + 31) / 32;     // sums, in groups of 32
    // A lane's 8 S products of a sum run as one chain of adds for short K and as two beyond, or their rounding shows (768 x 3072
    // against fp64: 1.9e-7 with one chain, 1.4e-7 with two, as the tensor-core kernel).
    constexpr int CHAINS = S > 3 ? 2 : 1;
    extern __shared__ __align__(16) float rw_smem[];
    const int steps = p.steps, KP = steps * RW_STEP;
    float* xs = rw_smem;                             // [M][KP], each step stored as [half][lane][4]
    __nv_bfloat16* gs = reinterpret_cast<__nv_bfloat16*>(xs + (size_t)M * KP);   // [KP] gain of the RMS norm
    float* ss = reinterpret_cast<float*>(gs + KP);   // [M][steps] pieces of the rows' sums of squares
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int groups = (p.N + R - 1) / R, stride = gridDim.x * RW_WARPS;
    int g = warp * gridDim.x + blockIdx.x;           // (neighbouring groups on different SMs)

    uint4 w[NT][R][S];
    auto load_rows = [&](int grp) {
#pragma unroll
        for (int t = 0; t < NT; ++t)
#pragma unroll
            for (int rr = 0; rr < R; ++rr) {
                const __nv_bfloat16* src = (t == 0 ? p.W : p.W2) + (size_t)min(grp * R + rr, p.N - 1) * p.K + lane * 8;
#pragma unroll
                for (int s = 0; s < S; ++s)
                    w[t][rr][s] = s < steps && s * RW_STEP + lane * 8 < p.K ? ldg_stream(src + s * RW_STEP) : make_uint4(0, 0, 0, 0);
            }
    };
    if (g < groups) load_rows(g);                    // weights and gain do not depend on the kernel before this one
    if (p.gain)
        for (int k = tid * 8; k < p.K; k += RW_THREADS * 8)
            *reinterpret_cast<uint4*>(gs + k) = *reinterpret_cast<const uint4*>(p.gain + k);
    if (p.m < M || KP > p.K)                         // rows past the block and the tail of K
        for (int i = tid * 4; i < M * KP; i += RW_THREADS * 4) *reinterpret_cast<float4*>(xs + i) = make_float4(0.f, 0.f, 0.f, 0.f);
    pdl_wait();
    pdl_trigger();
    if (GATHER) clear_words<RW_THREADS>(p.tickets, p.n_clear);   // (the first launch of a forward)
    __syncthreads();

    // ---- the block's rows: task (row, step) to a warp, four tasks' loads in flight; then each lane scales what it
    //      copied itself and takes the sums of squares
    const int tasks = p.m * steps;
#pragma unroll 4
    for (int t = warp; t < tasks; t += RW_WARPS) {
        const int r = t / steps, k = (t - r * steps) * RW_STEP;
        if (k + lane * 8 < p.K) {
            float* dst = xs + (size_t)r * KP + k + lane * 4;
            if (GATHER) {
                // The first projection of a forward gathers its rows itself (the first CTA also leaves them in fp32 for the
                // residual), a launch less: one row of the 68M shape 39.5 -> 38.3 us, five of the tiny draft 17.3 -> 16.3.  (As
                // a branch in every launch it cost the 60 launches of a t5-base-shaped forward 2 %.)
                int id = p.tokens[r];
                if (id < 0 || id >= p.vocab) {
                    if (blockIdx.x == 0 && lane == 0) set_status(p.status, CSD_ERR_BAD_TOKEN);
                    id = 0;
                }
                const uint4 e = *reinterpret_cast<const uint4*>(p.embed + (size_t)id * p.K + k + lane * 8);
                const float4 a = make_float4(bf16lo(e.x), bf16hi(e.x), bf16lo(e.y), bf16hi(e.y));
                const float4 b = make_float4(bf16lo(e.z), bf16hi(e.z), bf16lo(e.w), bf16hi(e.w));
                *reinterpret_cast<float4*>(dst) = a;
                *reinterpret_cast<float4*>(dst + 128) = b;
                if (blockIdx.x == 0) {
                    float* out = p.x_out + (size_t)r * p.ldx + k + lane * 8;
                    *reinterpret_cast<float4*>(out) = a;
                    *reinterpret_cast<float4*>(out + 4) = b;
                }
            } else {
                const float* src = p.X + (size_t)r * p.ldx + k + lane * 8;
                *reinterpret_cast<float4*>(dst) = *reinterpret_cast<const float4*>(src);
                *reinterpret_cast<float4*>(dst + 128) = *reinterpret_cast<const float4*>(src + 4);
            }
        }
    }
    if (p.gain) {
#pragma unroll 2
        for (int t = warp; t < tasks; t += RW_WARPS) {
            const int r = t / steps, k = (t - r * steps) * RW_STEP;
            float* dst = xs + (size_t)r * KP + k + lane * 4;
            float4 a = *reinterpret_cast<float4*>(dst), b = *reinterpret_cast<float4*>(dst + 128);
            float sq = (a.x * a.x + a.y * a.y + a.z * a.z + a.w * a.w) + (b.x * b.x + b.y * b.y + b.z * b.z + b.w * b.w);
            if (k + lane * 8 < p.K) {
                const uint4 gn = *reinterpret_cast<const uint4*>(gs + k + lane * 8);
                a.x *= bf16lo(gn.x); a.y *= bf16hi(gn.x); a.z *= bf16lo(gn.y); a.w *= bf16hi(gn.y);
                b.x *= bf16lo(gn.z); b.y *= bf16hi(gn.z); b.z *= bf16lo(gn.w); b.w *= bf16hi(gn.w);
                *reinterpret_cast<float4*>(dst) = a;
                *reinterpret_cast<float4*>(dst + 128) = b;
            }
            sq = warp_sum(sq);
            if (lane == 0) ss[t] = sq;
        }
    }
    // residual values this warp's first sums are added to travel meanwhile
    auto row_of = [&](int v) { return v % M; };
    auto col_of = [&](int v, int grp) { return grp * R + v / M; };
    float old[Q];
    auto load_old = [&](int grp) {
#pragma unroll
        for (int c = 0; c < Q; ++c) {
            const int v = c * 32 + lane;
            old[c] = p.epilogue == EPI_ADD && v < V && row_of(v) < p.m && col_of(v, grp) < p.N
                         ? p.Y[(size_t)row_of(v) * p.ldy + col_of(v, grp)] : 0.f;
        }
    };
    if (g < groups) load_old(g);
    __syncthreads();

#pragma unroll 1
    while (g < groups) {
        float acc[NT][V], acc2[NT][V];
#pragma unroll
        for (int t = 0; t < NT; ++t)
#pragma unroll
            for (int v = 0; v < V; ++v) acc[t][v] = acc2[t][v] = 0.f;
#pragma unroll
        for (int s = 0; s < S; ++s) {
            if (s >= steps) break;
            const float* xp = xs + s * RW_STEP + lane * 4;
#pragma unroll
            for (int r = 0; r < M; ++r) {
                const float4 xa = *reinterpret_cast<const float4*>(xp + (size_t)r * KP);
                const float4 xb = *reinterpret_cast<const float4*>(xp + (size_t)r * KP + 128);
#pragma unroll
                for (int t = 0; t < NT; ++t)
#pragma unroll
                    for (int rr = 0; rr < R; ++rr) {
                        const uint4 u = w[t][rr][s];
                        float d = acc[t][rr * M + r];
                        d = fmaf(bf16lo(u.x), xa.x, d); d = fmaf(bf16hi(u.x), xa.y, d);
                        d = fmaf(bf16lo(u.y), xa.z, d); d = fmaf(bf16hi(u.y), xa.w, d);
                        float e = CHAINS > 1 ? acc2[t][rr * M + r] : d;
                        e = fmaf(bf16lo(u.z), xb.x, e); e = fmaf(bf16hi(u.z), xb.y, e);
                        e = fmaf(bf16lo(u.w), xb.z, e); e = fmaf(bf16hi(u.w), xb.w, e);
                        acc[t][rr * M + r] = CHAINS > 1 ? d : e;
                        if (CHAINS > 1) acc2[t][rr * M + r] = e;
                    }
            }
        }
        if (CHAINS > 1) {
#pragma unroll
            for (int t = 0; t < NT; ++t)
#pragma unroll
                for (int v = 0; v < V; ++v) acc[t][v] += acc2[t][v];
        }
        const int cur = g;
        g += stride;
        if (g < groups) load_rows(g);                // in flight while this group is reduced and stored
#pragma unroll
        for (int c = 0; c < Q; ++c) {
            constexpr int W32 = V < 32 ? V : 32;
            float sum[NT];
#pragma unroll
            for (int t = 0; t < NT; ++t) {
                float part[W32];
#pragma unroll
                for (int i = 0; i < W32; ++i) part[i] = c * 32 + i < V ? acc[t][c * 32 + i < V ? c * 32 + i : 0] : 0.f;
                sum[t] = lane_sums<W32>(part, lane);
            }
            const int v = c * 32 + lane, r = row_of(v), n = col_of(v, cur);
            if (v < V && r < p.m && n < p.N) {
                float scale = 1.f;
                if (p.gain) {
                    float sq = 0.f;
                    for (int s = 0; s < steps; ++s) sq += ss[r * steps + s];
                    scale = 1.f / sqrtf(sq / (float)p.K + p.eps);
                }
                float val = sum[0] * scale;
                if (DUAL) val = (p.epilogue == EPI_GEGLU ? gelu_tanh(val) : silu(val)) * (sum[NT - 1] * scale);
                p.Y[(size_t)r * p.ldy + n] = val + old[c];
            }
        }
        if (g < groups) load_old(g);
    }
}

template <int M, int R, int S, bool DUAL, bool GATHER>
static csd_status launch_row_one(const RowParams& rp, cudaStream_t st) {
    auto kern = row_gemm_kernel<M, R, S, DUAL, GATHER>;
    static PerDevice ready;   // per instantiation
    const csd_status ok = allow_smem(ready, kern, RW_SMEM_MAX);
    if (ok != CSD_OK) return ok;
    const int groups = (rp.N + R - 1) / R;
    int grid = (groups + RW_WARPS - 1) / RW_WARPS;
    if (grid > 2 * tc_sm_count()) grid = 2 * tc_sm_count();
    PdlLaunch L(dim3((unsigned)grid), dim3(RW_THREADS), row_smem(M, rp.steps), st);
    CSD_CUDA(cudaLaunchKernelEx(&L.cfg, kern, rp));
    count_launch();
    return CSD_OK;
}

template <int M, int R, int S, bool DUAL>
static csd_status launch_row(const RowParams& rp, cudaStream_t st) {
    if (!DUAL && rp.tokens) return launch_row_one<M, R, S, DUAL, !DUAL>(rp, st);
    return launch_row_one<M, R, S, DUAL, false>(rp, st);
}

// Rows a warp takes at a time: one while the chip's 2368 resident warps can have a row each (spread
// over all SMs, shortest reduction), else as many as the registers hold.
template <int M, bool DUAL>
static csd_status launch_row_m(const RowParams& rp, cudaStream_t st) {
    if (!DUAL && rp.steps > 3) return launch_row<M, 1, RW_MAX_STEPS, false>(rp, st);
    if (rp.N <= 2 * RW_WARPS * tc_sm_count()) return launch_row<M, 1, 3, DUAL>(rp, st);
    return launch_row<M, (DUAL || M > 5 ? 2 : 4), 3, DUAL>(rp, st);
}

csd_status launch_linear_row(const LinearArgs& a, cudaStream_t st) {
    const bool dual = a.W2 != nullptr;
    if (!row_supported(a.m, a.N, a.K, dual)) return CSD_ERR_UNSUPPORTED;
    RowParams rp;
    rp.W = a.W; rp.W2 = a.W2; rp.X = a.X; rp.gain = a.gain; rp.Y = a.Y; rp.N = a.N; rp.K = a.K; rp.ldx = a.ldx; rp.ldy = a.ldy;
    rp.tokens = a.tokens; rp.embed = a.embed; rp.x_out = a.x_out; rp.vocab = a.vocab; rp.status = a.tokens ? status_word_device() : nullptr;
    rp.tickets = a.tickets; rp.n_clear = a.n_clear;
    rp.m = a.m; rp.steps = (a.K + RW_STEP - 1) / RW_STEP; rp.epilogue = a.epilogue; rp.eps = a.eps;
#define CSD_ROW_CASE(MM) case MM: return dual ? launch_row_m<MM, true>(rp, st) : launch_row_m<MM, false>(rp, st);
    switch (row_m(a.m)) {
        CSD_ROW_CASE(1) CSD_ROW_CASE(2) CSD_ROW_CASE(3) CSD_ROW_CASE(4) CSD_ROW_CASE(5) CSD_ROW_CASE(6) CSD_ROW_CASE(8)
    }
#undef CSD_ROW_CASE
    return CSD_ERR_INVALID_ARG;
}

}  // namespace csd
