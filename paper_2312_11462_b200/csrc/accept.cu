// Review rule of speculative sampling (Section 2; lenience / greedy: Section 3.1): one kernel while the
// rows are resident at once (accept_row_kernel), else three kernels over the vocabulary:
//   stats    one streaming pass over all (2k+1) logit vectors of every row: per 8192-logit piece
//            the max, arg-max and sum of exponentials (fp32).  This is the HBM-bound part: a
//            warp owns a piece, keeps 8 x 16 bytes per lane in flight with the next 8 already
//            requested, and needs no block-wide synchronisation.
//   decide   per row: merge the pieces, run the accept tests of all positions in parallel with
//            the Philox uniforms, find the first rejection n.
//   resample (temperature > 0 only) per row, at position n only, in fp64 so that the chosen token
//            does not depend on summation order or on fp32 rounding: the sums of both laws'
//            exponentials (the normalisers) and the mass of the residual max(0, p - q) (or of p after
//            k acceptances), by a cluster of CTAs a row or, beyond V = 65536, by chunks in one pass and
//            a kernel that takes the inverse-CDF pick from their sums.  exp() here is a short fp64 routine of this file (exp_neg), and no
//            law is normalised: every comparison is made on products instead of quotients.
#include "accept_layout.cuh"
#include "model.cuh"
#include "philox.cuh"
#include <math.h>
#include <mutex>

namespace csd {

constexpr int ST_THREADS = 256;
constexpr int ST_SUB = 1024;     // logits a warp has in registers at a time (8 x float4 per lane)
constexpr int RS_THREADS = 256;

enum : int { MODE_DONE = 0, MODE_RESID_LOGITS = 1, MODE_RESID_POINT = 2, MODE_TARGET_ONLY = 3 };

// ---------------------------------------------------------------------------------------------
// stats pass: grid-stride loop of warps over (vector, piece) items
// ---------------------------------------------------------------------------------------------
template <bool VEC>
__device__ __forceinline__ void load_sub(const float* __restrict__ src, int e0, int V, int lane, float (&v)[32]) {
    if (VEC) {
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const int e = e0 + 4 * (lane + 32 * j);
            float4 f = make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
            if (e < V) f = __ldcs(reinterpret_cast<const float4*>(src + e));
            v[4 * j + 0] = f.x; v[4 * j + 1] = f.y; v[4 * j + 2] = f.z; v[4 * j + 3] = f.w;
        }
    } else {
#pragma unroll
        for (int j = 0; j < 32; ++j) {
            const int e = e0 + lane + 32 * j;
            v[j] = e < V ? __ldcs(src + e) : -INFINITY;
        }
    }
}
template <bool VEC> __device__ __forceinline__ int sub_index(int e0, int lane, int j) {
    return VEC ? e0 + 4 * (lane + 32 * (j >> 2)) + (j & 3) : e0 + lane + 32 * j;
}

template <bool VEC>
__global__ void __launch_bounds__(ST_THREADS, 2)
accept_stats_kernel(const float* __restrict__ tl, const float* __restrict__ dl, long long n_tvec, int V,
                    float invT, int greedy, StatPartial* __restrict__ out, int nchunk, long long items) {
    pdl_wait();            // the logits come from the kernel before this one on the stream
    pdl_trigger();
    const int lane = threadIdx.x & 31;
    const long long warps = (long long)gridDim.x * (ST_THREADS / 32);
    for (long long item = (long long)blockIdx.x * (ST_THREADS / 32) + (threadIdx.x >> 5); item < items; item += warps) {
        const long long vec = item / nchunk;
        const int chunk = (int)(item % nchunk);
        const float* src = vec < n_tvec ? tl + vec * (long long)V : dl + (vec - n_tvec) * (long long)V;
        const int base = chunk * ST_CHUNK;
        const int nsub = (min(V, base + ST_CHUNK) - base + ST_SUB - 1) / ST_SUB;
        float mx = -INFINITY, sum = 0.f;
        int arg = 0x7fffffff;
        float cur[32], nxt[32];
        load_sub<VEC>(src, base, V, lane, cur);
        for (int s = 0; s < nsub; ++s) {
            const int e0 = base + s * ST_SUB;
            if (s + 1 < nsub) load_sub<VEC>(src, e0 + ST_SUB, V, lane, nxt);     // in flight while this batch is reduced
            // batch max with the smallest index attaining it (indices grow with j inside a lane)
            float bm = -INFINITY;
            int ba = 0x7fffffff;
#pragma unroll
            for (int j = 0; j < 32; ++j)
                if (cur[j] > bm) { bm = cur[j]; ba = sub_index<VEC>(e0, lane, j); }
            if (bm > mx) {          // later batches hold larger indices, so ">" keeps the earliest arg-max
                sum = mx > -INFINITY ? sum * __expf((mx - bm) * invT) : 0.f;
                mx = bm; arg = ba;
            }
            if (!greedy && mx > -INFINITY) {
                float a = 0.f;
#pragma unroll
                for (int j = 0; j < 32; ++j) a += __expf((cur[j] - mx) * invT);
                sum += a;
            }
            if (s + 1 < nsub) {
#pragma unroll
                for (int j = 0; j < 32; ++j) cur[j] = nxt[j];
            }
        }
        // lanes -> warp
        float wm = mx;
        int wa = arg;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const float om = __shfl_xor_sync(0xffffffffu, wm, o);
            const int oa = __shfl_xor_sync(0xffffffffu, wa, o);
            if (om > wm || (om == wm && oa < wa)) { wm = om; wa = oa; }
        }
        float scaled = (!greedy && mx > -INFINITY) ? sum * __expf((mx - wm) * invT) : 0.f;
        scaled = warp_sum(scaled);
        if (lane == 0) {
            StatPartial p;
            p.mx = wm; p.sum = scaled; p.arg = wa; p.pad = 0;
            out[item] = p;
        }
    }
}

// ---------------------------------------------------------------------------------------------
// decide pass: one CTA per row
// ---------------------------------------------------------------------------------------------
constexpr int MAX_K = 64;

// exp(x) for x <= 0 in fp64 by table and polynomial: x = (64 m + j) ln2/64 + r with |r| <= ln2/128,
// exp(x) = 2^m * 2^(j/64) * e^r; the 64 table entries are correctly rounded doubles made on the host,
// e^r is its Taylor series to r^5 (remainder below 4e-17), 2^m goes through the exponent field.
// Relative error about 3e-16.  Below -708 the result is 0 (under the smallest normal number).
__constant__ double c_exp2_table[64];
__device__ __forceinline__ void exp_table_to_shared(double* s_tab) {
    for (int i = threadIdx.x; i < 64; i += blockDim.x) s_tab[i] = c_exp2_table[i];
    __syncthreads();
}
// The rounding to n goes through the magic constant 1.5 * 2^52 (n is the low word of the sum): rint and the
// conversion to int run at a quarter of the fp64 rate and bounded the resample passes.
__device__ __forceinline__ double exp_neg(double x, const double* __restrict__ s_tab) {
    const double magic = 6755399441055744.0;
    const double t = fma(x, 92.33248261689366, magic);        // 64 / ln 2
    const double nf = t - magic;
    const int n = __double2loint(t);
    double r = fma(-nf, 0.01083042468962958, x);              // ln 2 / 64, high part (low 22 bits clear: nf * high is exact)
    r = fma(-nf, 6.619564634077006e-12, r);                   // ln 2 / 64, low part
    double p = 1.0 / 120.0;
    p = fma(p, r, 1.0 / 24.0);
    p = fma(p, r, 1.0 / 6.0);
    p = fma(p, r, 0.5);
    p = fma(p, r, 1.0);
    p *= r;                                                   // e^r - 1
    const double tj = s_tab[n & 63];
    const double v = fma(tj, p, tj);
    const int hi = __double2hiint(v) + ((n >> 6) << 20);      // m >= -1022: stays a normal number
    return x > -708.0 ? __hiloint2double(hi, __double2loint(v)) : 0.0;
}

// u q(x) < l p(x) without a division; no lenience for the statistical drafter's tokens (Appendix B)
__device__ __forceinline__ bool accept_test(double u, float tx, float mt, float zt, bool point, float dx, float mq, float zq,
                                            double inv_temp, float lenience, const double* __restrict__ s_tab) {
    const double ep = exp_neg(((double)tx - (double)mt) * inv_temp, s_tab);
    if (point) return u * (double)zt < ep;
    const double eq = exp_neg(((double)dx - (double)mq) * inv_temp, s_tab);
    return u * eq * (double)zt < (double)lenience * ep * (double)zq;
}

// a later piece (larger indices) joins the running (max, sum, arg-max)
__device__ __forceinline__ void merge_stat(float& mx, float& z, int& arg, const StatPartial& q, float invT) {
    if (q.mx > mx) {
        z = (mx > -INFINITY ? z * __expf((mx - q.mx) * invT) : 0.f) + q.sum;
        mx = q.mx; arg = q.arg;
    } else if (q.mx > -INFINITY) {
        z += q.sum * __expf((q.mx - mx) * invT);
    }
}

// the pieces held by G neighbouring lanes, in index order, into the first of them
template <int G>
__device__ __forceinline__ void merge_stat_lanes(StatPartial& a, float invT) {
#pragma unroll
    for (int o = 1; o < G; o <<= 1) {
        StatPartial q;
        q.mx = __shfl_down_sync(0xffffffffu, a.mx, o); q.sum = __shfl_down_sync(0xffffffffu, a.sum, o);
        q.arg = __shfl_down_sync(0xffffffffu, a.arg, o); q.pad = 0;
        if (((int)threadIdx.x & (2 * o - 1)) == 0) merge_stat(a.mx, a.sum, a.arg, q, invT);
    }
}

constexpr int DC_THREADS = 512, DC_LANES = 16;   // lanes that merge one vector's pieces

__global__ void __launch_bounds__(DC_THREADS)
accept_decide_kernel(const float* __restrict__ tl, const float* __restrict__ dl, const int* __restrict__ onehot,
                     const int* __restrict__ tokens, int rows, int k, int V, float temperature, float lenience,
                     uint64_t seed, uint64_t step, const StatPartial* __restrict__ part, int nchunk,
                     int* __restrict__ n_acc, int* __restrict__ out_tok, RowInfo* __restrict__ info,
                     unsigned* __restrict__ tickets, int* status) {
    const int row = blockIdx.x, tid = threadIdx.x;
    __shared__ float s_mx[2 * MAX_K + 1];
    __shared__ float s_z[2 * MAX_K + 1];
    __shared__ int s_arg[2 * MAX_K + 1];
    __shared__ int s_acc[MAX_K], s_x[MAX_K], s_point[MAX_K];
    __shared__ double s_u2[MAX_K], s_tab[64];
    const bool greedy = temperature == 0.f;
    const float invT = greedy ? 1.f : 1.f / temperature;
    if (!greedy && tid < 64) s_tab[tid] = c_exp2_table[tid];
    pdl_wait();
    pdl_trigger();
    const int nvec_row = dl ? 2 * k + 1 : k + 1;
    const long long n_tvec = (long long)rows * (k + 1);
    // what the accept tests need besides the statistics travels while those are merged (thread i: position i)
    int x = 0;
    bool bad = false, point = true;
    float tx = 0.f, dx = 0.f;
    if (tid < k) {
        x = tokens[(long long)row * k + tid];
        bad = x < 0 || x >= V;
        point = dl == nullptr || (onehot && onehot[(long long)row * k + tid] != 0);
        if (!greedy && !bad) {
            tx = tl[((long long)row * (k + 1) + tid) * V + x];
            if (!point) dx = dl[((long long)row * k + tid) * V + x];
        }
    }
    // ---- merge the pieces of every vector of this row: 16 lanes a vector, so that a piece per lane is requested at
    //      once (one thread per vector walked 16 pieces of V = 128256 in four round trips)
    for (int i0 = 0; i0 < nvec_row; i0 += DC_THREADS / DC_LANES) {
        const int i = i0 + tid / DC_LANES, l = tid % DC_LANES;
        StatPartial a;
        a.mx = -INFINITY; a.sum = 0.f; a.arg = 0x7fffffff; a.pad = 0;
        if (i < nvec_row) {
            const long long vec = i <= k ? (long long)row * (k + 1) + i : n_tvec + (long long)row * k + (i - k - 1);
            const StatPartial* p = part + vec * nchunk;
            const int each = (nchunk + DC_LANES - 1) / DC_LANES;      // a lane's pieces are neighbours, in index order
            for (int c = l * each; c < min(nchunk, (l + 1) * each); ++c) merge_stat(a.mx, a.sum, a.arg, p[c], invT);
        }
        merge_stat_lanes<DC_LANES>(a, invT);
        if (i < nvec_row && l == 0) { s_mx[i] = a.mx; s_z[i] = a.sum; s_arg[i] = a.arg; }
    }
    if (tid == 0 && tickets) tickets[row] = 0u;        // for the resample's CTAs of a row
    __syncthreads();
    RowInfo ri;
    ri.n = k; ri.mode = MODE_DONE; ri.x = 0; ri.pad = 0; ri.max_t = 0; ri.max_q = 0; ri.u2 = 0; ri.z_t = ri.z_q = 1.f;
    if (tid < k) {                              // a drafted id outside the vocabulary is rejected and recorded
        if (bad) set_status(status, CSD_ERR_BAD_TOKEN);
        s_x[tid] = bad ? 0 : x; s_point[tid] = point ? 1 : 0;
        if (greedy) s_acc[tid] = x == s_arg[tid];
    }
    const uint32_t k0 = (uint32_t)seed, k1 = (uint32_t)(seed >> 32);
    const uint32_t c2 = (uint32_t)step, c3 = (uint32_t)(step >> 32);
    // ---- the accept tests of all positions at once (thread i: position i)
    if (!greedy && tid < k) {
        const Philox4 r = philox4x32_10((uint32_t)tid, (uint32_t)row, c2, c3, k0, k1);
        const double inv_temp = 1.0 / (double)temperature;
        s_acc[tid] = !bad && accept_test(word_uniform(r.w[0]), tx, s_mx[tid], s_z[tid], point, dx, point ? 0.f : s_mx[k + 1 + tid],
                                         point ? 1.f : s_z[k + 1 + tid], inv_temp, lenience, s_tab);
        s_u2[tid] = word_uniform(r.w[1]);
    }
    __syncthreads();
    if (tid != 0) return;
    int n = 0;
    while (n < k && s_acc[n]) ++n;
    if (greedy) {
        out_tok[row] = s_arg[n];
    } else if (n < k) {
        ri.mode = s_point[n] ? MODE_RESID_POINT : MODE_RESID_LOGITS;
        ri.x = s_x[n];
        ri.max_t = (double)s_mx[n];
        ri.max_q = s_point[n] ? 0.0 : (double)s_mx[k + 1 + n];
        ri.u2 = s_u2[n];
        ri.z_t = s_z[n]; ri.z_q = s_point[n] ? 1.f : s_z[k + 1 + n];
    } else {
        const Philox4 r = philox4x32_10((uint32_t)k, (uint32_t)row, c2, c3, k0, k1);
        ri.mode = MODE_TARGET_ONLY;
        ri.max_t = (double)s_mx[k];
        ri.u2 = word_uniform(r.w[1]);
    }
    ri.n = n;
    n_acc[row] = n;
    info[row] = ri;
}

// ---------------------------------------------------------------------------------------------
// resample passes (fp64) of long vocabularies: sums, then the pick.  In the first a WARP owns a chunk of a row (two sets of 512 logits,
// or eight where the scratch is small; 8 neighbours a lane and load); no block-wide synchronisation.  The residual max(0, p - q) needs
// both normalisers, which are known when every entry has been seen; but which entries it keeps is known before that for all but a
// few, from the fp32 sums of the stats pass and a bound on their error.  So one pass sums, per chunk, both laws' exponentials (the
// normalisers) and, apart, those of the entries that stay: a chunk's residual mass is then A Zq - B Zp, plus the few undecided
// entries, which are listed and taken up by the second kernel; it reads a row's sums, not its logits, but for the chunk it picks
// from and for chunks with more undecided entries than a list holds, which it forms anew.
// Bound by the fp64 pipe (about 13 instructions an exponential).  Against a pass for the normalisers and one for the masses of all
// entries (31 and 47 us at 64 rows, V = 128256), us a call: 64 rows, k = 16 245 -> 217, k = 4 122 -> 92; 16 rows, k 8, V 98315
// 63.5 -> 45.0; 2 rows, k 15 38.6 -> 29.0.  Laws that nearly agree have full lists throughout (logits apart by 0.005 and less, 64 rows
// 109 -> 106 to 112, 20 rows 54 -> 49 to 53): formed by one warp a row they took 1090 and 940, by the warps that had
// summed them, staying for the normalisers, 187 and 96.  Three blocks an SM: with two, 64 rows, k = 16 222.
// Every sum has one fixed order: a lane's entries, lanes by xor-shuffle or prefix scan, chunks in index order.
// ---------------------------------------------------------------------------------------------
constexpr unsigned short RS_NONE = 0xffff, RS_FULL = 0xfffe;
// Distance of the laws' logarithms within which an entry is undecided.  The fp32 sums are off by at most the terms' own errors (2 ulp
// of __expf, 1.2 more for each unit of the exponent, whose mean under a law is below ln V) and 300 roundings: 2e-5 each; the
// comparison itself by 2^-23 of the exponents.
constexpr float RS_BAND = 5e-5f;

// eight consecutive logits of a vector (two 16-byte loads when the vector allows it); past V: -inf
__device__ __forceinline__ void load8(const float* __restrict__ src, int e0, int V, bool vec, float (&v)[8]) {
    if (vec && e0 + 7 < V) {
        const float4 a = __ldcs(reinterpret_cast<const float4*>(src + e0));
        const float4 b = __ldcs(reinterpret_cast<const float4*>(src + e0 + 4));
        v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w; v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
    } else {
#pragma unroll
        for (int j = 0; j < 8; ++j) v[j] = e0 + j < V ? __ldcs(src + e0 + j) : -INFINITY;
    }
}

// The residual max(0, p - q) of an entry up to a positive factor that is the same for the whole row (the pick
// compares sums with u2 times their total): Zp Zq (et / Zp - ed / Zq) for two laws, Zp (et / Zp - [e == x]) against
// a point mass, et for the target law itself.  et and ed are exp((logit - max) / T).
__device__ __forceinline__ double residual_from(int mode, double et, double ed, double Zp, double Zq, bool at_x) {
    if (mode == MODE_TARGET_ONLY) return et;
    const double a = mode == MODE_RESID_POINT ? et : et * Zq;
    const double b = mode == MODE_RESID_POINT ? (at_x ? Zp : 0.0) : ed * Zp;
    return a > b ? a - b : 0.0;
}

struct ResidualCtx {
    const float* t; const float* d; const double* tab;
    double max_t, max_q, invT, Zp, Zq;
    int mode, x;
};
__device__ __forceinline__ ResidualCtx residual_ctx(const RowInfo& ri, int row, const float* tl, const float* dl, int k, int V, float temperature,
                                                    const double* tab) {
    ResidualCtx c;
    c.t = tl + ((long long)row * (k + 1) + ri.n) * V;
    c.d = ri.mode == MODE_RESID_LOGITS ? dl + ((long long)row * k + ri.n) * V : nullptr;
    c.tab = tab;
    c.max_t = ri.max_t; c.max_q = ri.max_q; c.invT = 1.0 / (double)temperature; c.Zp = c.Zq = 0.0;
    c.mode = ri.mode; c.x = ri.x;
    return c;
}
__device__ __forceinline__ bool residual_vec(const ResidualCtx& c, int V) {      // 16-byte loads
    return (V % 4 == 0) && ((((uintptr_t)c.t) & 15) == 0) && (!c.d || (((uintptr_t)c.d) & 15) == 0);
}
__device__ __forceinline__ double residual_of(const ResidualCtx& c, int e, float tv, float dv) {
    const double et = exp_neg(((double)tv - c.max_t) * c.invT, c.tab);
    const double ed = c.mode == MODE_RESID_LOGITS ? exp_neg(((double)dv - c.max_q) * c.invT, c.tab) : 0.0;
    return residual_from(c.mode, et, ed, c.Zp, c.Zq, e == c.x);
}

__device__ __forceinline__ double warp_scan(double v, int lane) {      // inclusive prefix
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const double up = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += up;
    }
    return v;
}
__global__ void __launch_bounds__(RS_THREADS, 3)
resample_sums_kernel(const float* __restrict__ tl, const float* __restrict__ dl, int rows, int k, int V, float temperature,
                     const RowInfo* __restrict__ info, ChunkSums* __restrict__ sums, unsigned short* __restrict__ lists, int nchunk, int sets) {
    __shared__ double s_tab[64];
    exp_table_to_shared(s_tab);
    pdl_wait();            // the row records come from the decide pass
    pdl_trigger();
    const int lane = threadIdx.x & 31;
    const long long item = (long long)blockIdx.x * (blockDim.x / 32) + (threadIdx.x >> 5);
    const int row = (int)(item / nchunk), chunk = (int)(item % nchunk);
    if (row >= rows) return;
    const RowInfo ri = info[row];
    const ResidualCtx c = residual_ctx(ri, row, tl, dl, k, V, temperature, s_tab);
    const bool vec = residual_vec(c, V);
    unsigned short* list = lists + item * RS_LIST;
    const float fT = 1.f / temperature, edge = c.d ? logf(ri.z_t) - logf(ri.z_q) : 0.f;   // stays: x_t - x_d > edge
    const float mt = (float)ri.max_t, mq = (float)ri.max_q;
    ChunkSums acc{0.0, 0.0, 0.0, 0.0};
    int listed = 0;
    float nt[8], nd[8];
    load8(c.t, chunk * sets * RS_CHUNK + lane * 8, V, vec, nt);
    if (c.d) load8(c.d, chunk * sets * RS_CHUNK + lane * 8, V, vec, nd);
#pragma unroll 1
    for (int half = 0; half < 2 * sets; ++half) {
        const int at = (chunk * sets * 2 + half) * 256 + lane * 8;
        float tv[8], dv[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) { tv[j] = nt[j]; dv[j] = nd[j]; }
        if (half + 1 < 2 * sets) {                                       // in flight while this half is summed
            load8(c.t, at + 256, V, vec, nt);
            if (c.d) load8(c.d, at + 256, V, vec, nd);
        }
        unsigned open = 0;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const double et = exp_neg(((double)tv[j] - c.max_t) * c.invT, s_tab);         // -inf (past V) gives 0
            acc.p += et;
            if (c.d) {
                const double ed = exp_neg(((double)dv[j] - c.max_q) * c.invT, s_tab);
                acc.q += ed;
                if (listed > RS_LIST) continue;                              // a full list: formed anew in any case
                const float over = (tv[j] - mt) * fT - (dv[j] - mq) * fT - edge;
                const float band = RS_BAND + 3e-7f * (fabsf((tv[j] - mt) * fT) + fabsf((dv[j] - mq) * fT));
                const bool stays = over > band || dv[j] == -INFINITY;
                acc.a += stays ? et : 0.0;
                acc.b += stays ? ed : 0.0;
                // (also what does not compare: both laws without the entry, not-a-number)
                if (!stays && !(over < -band) && at + j < V && !(tv[j] == -INFINITY)) open |= 1u << j;
            } else {
                acc.a += at + j != c.x || c.mode != MODE_RESID_POINT ? et : 0.0;
            }
        }
        while (listed <= RS_LIST && __any_sync(0xffffffffu, open != 0)) {     // rare
            const unsigned who = __ballot_sync(0xffffffffu, open != 0);
            const int place = listed + __popc(who & ((1u << lane) - 1u));
            if (open && place < RS_LIST) list[place] = (unsigned short)(at + __ffs(open) - 1 - chunk * sets * RS_CHUNK);
            open &= open - 1;
            listed += __popc(who);
        }
    }
    acc.p = warp_sum(acc.p);
    if (c.d) { acc.q = warp_sum(acc.q); acc.b = warp_sum(acc.b); }
    acc.a = warp_sum(acc.a);
    __syncwarp();                                                        // (a lane's entry in list[0] before the mark there)
    if (lane == 0) {
        sums[item] = acc;
        if (listed > RS_LIST) list[0] = RS_FULL;
        else if (listed < RS_LIST) list[listed] = RS_NONE;
    }
}

// mass of the residual of two laws over one chunk, by a warp
__device__ __forceinline__ double chunk_mass(const ResidualCtx& c, int at, int end, int V, bool vec, int lane) {
    double sr = 0.0;
    float nt[8], nd[8];
    load8(c.t, at + lane * 8, V, vec, nt);
    load8(c.d, at + lane * 8, V, vec, nd);
#pragma unroll 1
    for (; at < end; at += 256) {
        float tv[8], dv[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) { tv[j] = nt[j]; dv[j] = nd[j]; }
        if (at + 256 < end) {                                                // in flight while these are summed
            load8(c.t, at + 256 + lane * 8, V, vec, nt);
            load8(c.d, at + 256 + lane * 8, V, vec, nd);
        }
#pragma unroll
        for (int j = 0; j < 8; ++j) sr += residual_of(c, at + lane * 8 + j, tv[j], dv[j]);
    }
    return warp_sum(sr);
}

// The normalisers, every chunk's mass into its b, the pick.  A row's first CTA does it, unless some of its chunks have full lists:
// then all `per_row` CTAs of the row form those anew, a warp a chunk, and the last of them to finish does the rest.
__global__ void __launch_bounds__(RS_THREADS, 3)
resample_pick_kernel(const float* __restrict__ tl, const float* __restrict__ dl, int k, int V, float temperature,
                     const RowInfo* __restrict__ info, ChunkSums* sums, const unsigned short* __restrict__ lists,
                     unsigned* __restrict__ tickets, int nchunk, int sets, int per_row, int* __restrict__ out_tok) {
    constexpr int WARPS = RS_THREADS / 32;
    __shared__ double s_tab[64], s_warp[2 * WARPS];
    __shared__ int s_int[2 * WARPS], s_chunk;
    __shared__ double s_cum;
    exp_table_to_shared(s_tab);
    pdl_wait();            // the chunks' sums come from the pass before this one
    pdl_trigger();
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, row = blockIdx.x / per_row, share = blockIdx.x % per_row;
    const RowInfo ri = info[row];
    ResidualCtx c = residual_ctx(ri, row, tl, dl, k, V, temperature, s_tab);
    const bool vec = residual_vec(c, V);
    const int len = sets * RS_CHUNK;                     // logits of a chunk
    ChunkSums* mine = sums + (long long)row * nchunk;
    auto words = [&](int ch) { return reinterpret_cast<const uint32_t*>(lists + ((long long)row * nchunk + ch) * RS_LIST); };
    auto is_full = [&](int ch) { return c.d && (words(ch)[0] & 0xffffu) == RS_FULL; };
    bool full = false;
    double sp = 0.0, sq = 0.0;
    for (int ch = tid; ch < nchunk; ch += RS_THREADS) {
        full = full || is_full(ch);
        sp += mine[ch].p; sq += mine[ch].q;
    }
    full = __syncthreads_or(full);
    if (share != 0 && !full) return;
    // ---- the normalisers (every CTA of the row adds the same numbers in the same order)
    sp = warp_sum(sp); sq = warp_sum(sq);
    if (lane == 0) { s_warp[warp] = sp; s_warp[WARPS + warp] = sq; }
    __syncthreads();
    sp = sq = 0.0;
#pragma unroll
    for (int w = 0; w < WARPS; ++w) { sp += s_warp[w]; sq += s_warp[WARPS + w]; }
    c.Zp = sp; c.Zq = sq;
    if (full) {
#pragma unroll 1
        for (int ch = share * WARPS + warp; ch < nchunk; ch += per_row * WARPS)
            if (is_full(ch)) {
                const double m = chunk_mass(c, ch * len, (ch + 1) * len, V, vec, lane);
                if (lane == 0) __stcg(&mine[ch].b, m);
            }
        if (per_row > 1) {
            __syncthreads();
            if (tid == 0) {
                __threadfence();
                s_chunk = (int)atomicAdd(&tickets[row], 1u);
                __threadfence();
            }
            __syncthreads();
            if (s_chunk != per_row - 1) return;
        }
    }
    // ---- the other chunks' masses: a thread a chunk
    if (c.mode != MODE_TARGET_ONLY)
        for (int ch = tid; ch < nchunk; ch += RS_THREADS) {
            if (is_full(ch)) continue;
            double mass = mine[ch].a;
            if (c.d) {
                mass = mass * c.Zq - mine[ch].b * c.Zp;
                float tv[RS_LIST], dv[RS_LIST];
                int at[RS_LIST], n = 0;
#pragma unroll
                for (int i = 0; i < RS_LIST; ++i) {
                    const unsigned e = (words(ch)[i / 2] >> (16 * (i & 1))) & 0xffffu;
                    if (n == i && e != RS_NONE) { at[i] = ch * len + (int)e; tv[i] = c.t[at[i]]; dv[i] = c.d[at[i]]; n = i + 1; }
                }
#pragma unroll
                for (int i = 0; i < RS_LIST; ++i)
                    if (i < n) mass += residual_of(c, at[i], tv[i], dv[i]);
            }
            __stcg(&mine[ch].b, mass > 0.0 ? mass : 0.0);                    // (rounding of the difference)
        }
    __syncthreads();
    // inclusive prefix over the CTA's threads; `total` of all
    auto block_scan = [&](double v, double& total) {
        const double in = warp_scan(v, lane);
        __syncthreads();
        if (lane == 31) s_warp[warp] = in;
        __syncthreads();
        double before = 0.0;
        total = 0.0;
#pragma unroll
        for (int w = 0; w < WARPS; ++w) {
            if (w == warp) before = total;
            total += s_warp[w];
        }
        return before + in;
    };
    // ---- which chunk holds u2 * S: a thread owns neighbouring chunks; a second time with the target law itself if the
    //      residual is empty.  Rounding may leave none, then the last chunk that carries mass.
    const int each = (nchunk + RS_THREADS - 1) / RS_THREADS, c_lo = min(nchunk, tid * each), c_hi = min(nchunk, c_lo + each);
    double own = 0.0, incl = 0.0, S = 0.0;
    auto mass_of = [&](int ch) -> double { return c.mode == MODE_TARGET_ONLY ? mine[ch].p : __ldcg(&mine[ch].b); };
#pragma unroll 1
    for (int pass = 0; pass < 2; ++pass) {
        own = 0.0;
        for (int ch = c_lo; ch < c_hi; ++ch) own += mass_of(ch);
        incl = block_scan(own, S);
        if (pass == 0 && c.mode != MODE_TARGET_ONLY && (!(S > 0.0) || !isfinite(S))) { c.mode = MODE_TARGET_ONLY; continue; }
        break;
    }
    const double target = ri.u2 * S;
    // first thread whose prefix exceeds the target, last thread with mass
    auto first_last = [&](bool past, bool some, int& first, int& last) {
        const unsigned a = __ballot_sync(0xffffffffu, past), z = __ballot_sync(0xffffffffu, some);
        if (lane == 0) { s_int[warp] = a ? warp * 32 + __ffs(a) - 1 : -1; s_int[WARPS + warp] = z ? warp * 32 + 31 - __clz(z) : -1; }
        __syncthreads();
        first = last = -1;
#pragma unroll
        for (int w = 0; w < WARPS; ++w) {
            if (first < 0) first = s_int[w];
            if (s_int[WARPS + w] >= 0) last = s_int[WARPS + w];
        }
        __syncthreads();
    };
    int first, last;
    first_last(incl > target, own > 0.0, first, last);
    const bool forced = first < 0;
    if (tid == (forced ? max(last, 0) : first)) {
        double cum = incl - own;
        int last_pos = c_lo, hit = -1;
        for (int ch = c_lo; ch < c_hi; ++ch) {
            const double m = mass_of(ch);
            if (m > 0.0) last_pos = ch;
            if (!forced && cum + m > target) { hit = ch; break; }
            cum += m;
        }
        if (hit < 0) {                                  // the last chunk with mass, from its own start
            hit = last_pos;
            cum = incl - own;
            for (int ch = c_lo; ch < last_pos; ++ch) cum += mass_of(ch);
        }
        s_chunk = hit; s_cum = cum;
    }
    __syncthreads();
    double cum = s_cum;
    const int begin = s_chunk * len, end = min(V, begin + len);
    // ---- the entry: smallest index whose cumulative mass exceeds the target, else the last that carries mass
    int pick = -1, carries = -1;
#pragma unroll 1
    for (int e = begin; e < end && pick < 0; e += RS_THREADS * 4) {
        const int at = e + tid * 4;
        double r[4], local = 0.0, total;
        int my_last = -1;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const bool in = at + j < end;
            r[j] = in ? residual_of(c, at + j, c.t[at + j], c.mode == MODE_RESID_LOGITS ? c.d[at + j] : 0.f) : 0.0;
            if (r[j] > 0.0) my_last = j;
            local += r[j];
        }
        double run = cum + (block_scan(local, total) - local);
        int found = -1;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            run += r[j];
            if (!forced && found < 0 && r[j] > 0.0 && run > target) found = j;
        }
        first_last(found >= 0, my_last >= 0, first, last);
        if (tid == first || tid == last) s_int[tid == first ? 0 : 1] = at + (tid == first ? found : my_last);
        if (tid == first && tid == last) s_int[1] = at + my_last;
        __syncthreads();
        if (first >= 0) pick = s_int[0];
        if (last >= 0) carries = s_int[1];
        __syncthreads();
        cum += total;
    }
    if (tid == 0) out_tok[row] = pick >= 0 ? pick : max(carries, 0);
}

// ---------------------------------------------------------------------------------------------
// resample, one kernel: a row is a thread-block cluster of up to RF_MAXC CTAs; a CTA keeps its
// slice of the two logit vectors (position n only) in registers, so global memory is read once.
// First exchange: per-CTA sums of the exponentials, exchanged through distributed shared memory (a lane per CTA) -> the
// normalisers.  Second exchange: per-CTA residual mass -> total mass S and the CTA whose slice holds
// u2 * S.  That CTA scans its threads' sums in thread order and picks the entry.  All sums have a
// fixed order (lanes by xor-shuffle or prefix scan, warps and CTAs in index order).
// ---------------------------------------------------------------------------------------------
constexpr int RF_THREADS = 512, RF_WARPS = RF_THREADS / 32, RF_PER = 16, RF_SLICE = RF_THREADS * RF_PER;
constexpr int RF_MAXC = 8;   // (clusters of 16 run one per GPC at a time: 64 rows, k 4, V 128256 199 us a call; the passes take 92)

__device__ __forceinline__ uint32_t cluster_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ void cluster_sync_all() {
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ double cluster_read_f64(const double* local, uint32_t rank) {
    uint32_t a = (uint32_t)__cvta_generic_to_shared(local), r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
    double v;
    asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(r) : "memory");
    return v;
}

// ALONE: a row of one CTA, which exchanges with nobody (barriers of a cluster of one and reads through its window: 200 rows, k 1,
// V 512 24.8 us a call, 21.9 so; asked at run time, larger clusters lose 1 to 2 %)
template <bool ALONE>
__global__ void __launch_bounds__(RF_THREADS, 1)
resample_fused_kernel(const float* __restrict__ tl, const float* __restrict__ dl, int k, int V, float temperature,
                      const RowInfo* __restrict__ info, int csize, int* __restrict__ out_tok) {
    const int row = blockIdx.x / csize;
    const uint32_t rank = cluster_rank();
    pdl_wait();            // the row records come from the decide pass
    pdl_trigger();
    const RowInfo ri = info[row];
    if (ri.mode == MODE_DONE) return;                 // (the same decision in every CTA of the cluster)
    __shared__ double s_warp[2 * RF_WARPS], s_ex[4];  // s_ex: this CTA's contributions to the exchanges
    __shared__ double s_tab[64];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    auto sync_row = [] { if (ALONE) __syncthreads(); else cluster_sync_all(); };
    auto read_of = [](const double* p, uint32_t r) { return ALONE ? *p : cluster_read_f64(p, r); };
    exp_table_to_shared(s_tab);
    const double invT = 1.0 / (double)temperature;
    const float* t = tl + ((long long)row * (k + 1) + ri.n) * V;
    const float* d = ri.mode == MODE_RESID_LOGITS ? dl + ((long long)row * k + ri.n) * V : nullptr;
    const int e0 = (int)rank * RF_SLICE + threadIdx.x * RF_PER;
    // ---- this thread's entries, read once; their exponentials stay in registers for both rounds (formed anew in the second one they
    //      let two CTAs share an SM, but the fp64 pipe is what a wave waits for: 64 rows, k 16, V 32000 78.8 -> 80.9 us, V 60000 24.8 -> 30.1)
    double et[RF_PER], ed[RF_PER];
    const bool vec = (V % 4 == 0) && ((((uintptr_t)t) & 15) == 0) && (!d || (((uintptr_t)d) & 15) == 0);
    double sp = 0.0, sq = 0.0;
#pragma unroll
    for (int j = 0; j < RF_PER; j += 4) {
        const int e = e0 + j;
        float tv[4], dv[4];
        if (vec && e + 3 < V) {
            const float4 a = __ldcs(reinterpret_cast<const float4*>(t + e));
            tv[0] = a.x; tv[1] = a.y; tv[2] = a.z; tv[3] = a.w;
            if (d) {
                const float4 b = __ldcs(reinterpret_cast<const float4*>(d + e));
                dv[0] = b.x; dv[1] = b.y; dv[2] = b.z; dv[3] = b.w;
            } else { dv[0] = dv[1] = dv[2] = dv[3] = -INFINITY; }
        } else {
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                tv[i] = e + i < V ? __ldcs(t + e + i) : -INFINITY;
                dv[i] = (d && e + i < V) ? __ldcs(d + e + i) : -INFINITY;
            }
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            et[j + i] = exp_neg(((double)tv[i] - ri.max_t) * invT, s_tab);   // -inf (past V) gives 0
            ed[j + i] = d ? exp_neg(((double)dv[i] - ri.max_q) * invT, s_tab) : 0.0;
            sp += et[j + i];
            sq += ed[j + i];
        }
    }
    // ---- first exchange: normalisers (lanes 0-15 hold the warps', then the CTAs' Zp, lanes 16-31 their Zq)
    auto half_sum = [](double a) {
#pragma unroll
        for (int o = RF_WARPS / 2; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
        return a;
    };
    sp = warp_sum(sp); sq = warp_sum(sq);
    if (lane == 0) { s_warp[warp] = sp; s_warp[RF_WARPS + warp] = sq; }
    __syncthreads();
    if (warp == 0) {
        const double a = half_sum(s_warp[lane]);
        if (lane % RF_WARPS == 0) s_ex[lane / RF_WARPS] = a;
    }
    sync_row();
    double Zp, Zq;
    {
        const double a = half_sum(lane % RF_WARPS < csize ? read_of(&s_ex[lane / RF_WARPS], (uint32_t)(lane % RF_WARPS)) : 0.0);
        Zp = __shfl_sync(0xffffffffu, a, 0); Zq = __shfl_sync(0xffffffffu, a, RF_WARPS);
    }
    const int xn = ri.x;
    // ---- second exchange: masses (a second time with the target law itself if the residual is empty)
    int mode = ri.mode, owner = 0;
    bool forced = false;
    double local = 0.0, run = 0.0, head = 0.0, target = 0.0;   // this thread's mass, the warps' up to lane, the CTAs' before this one
    auto resid = [&](int j) -> double { return e0 + j < V ? residual_from(mode, et[j], ed[j], Zp, Zq, e0 + j == xn) : 0.0; };
#pragma unroll 1
    for (int pass = 0; pass < 2; ++pass) {
        local = 0.0;
#pragma unroll
        for (int j = 0; j < RF_PER; ++j) local += resid(j);
        const double mass_w = warp_sum(local);
        __syncthreads();
        if (lane == 0) s_warp[warp] = mass_w;
        __syncthreads();
        run = warp_scan(lane < RF_WARPS ? s_warp[lane] : 0.0, lane);
        if (threadIdx.x == RF_WARPS - 1) s_ex[2 + pass] = run;
        sync_row();
        const double m = lane < csize ? read_of(&s_ex[2 + pass], (uint32_t)lane) : 0.0;
        const double incl = warp_scan(m, lane), total = __shfl_sync(0xffffffffu, incl, csize - 1);
        if (pass == 0 && mode != MODE_TARGET_ONLY && (!(total > 0.0) || !isfinite(total))) { mode = MODE_TARGET_ONLY; continue; }
        // the CTA whose masses reach past u2 * total; rounding may leave none, then the last one that carries mass
        target = ri.u2 * total;
        const unsigned past = __ballot_sync(0xffffffffu, lane < csize && incl > target);
        const unsigned some = __ballot_sync(0xffffffffu, m > 0.0);
        forced = past == 0;
        owner = past ? __ffs(past) - 1 : (some ? 31 - __clz(some) : 0);
        head = __shfl_sync(0xffffffffu, incl - m, (int)rank);
        break;
    }
    if (!ALONE) asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");     // this CTA has read what it needs of the others
    if ((int)rank == owner) {
        // ---- in it the warp, then the entry: the smallest index whose cumulative mass exceeds the target; forced, or where
        //      rounding leaves none: the last entry that carries mass
        const unsigned past = __ballot_sync(0xffffffffu, lane < RF_WARPS && head + run > target);
        const unsigned some = __ballot_sync(0xffffffffu, lane < RF_WARPS && s_warp[lane % RF_WARPS] > 0.0);
        const int wpick = past && !forced ? __ffs(past) - 1 : (some ? 31 - __clz(some) : 0);
        const double before = __shfl_sync(0xffffffffu, run, (wpick + 31) & 31);
        if (warp == wpick) {
            double cum = head + (wpick > 0 ? before : 0.0) + (warp_scan(local, lane) - local);
            int found = 0x7fffffff, my_last = -1;
#pragma unroll
            for (int j = 0; j < RF_PER; ++j) {
                const double r = resid(j);
                if (r > 0.0) my_last = e0 + j;
                cum += r;
                if (!forced && found == 0x7fffffff && r > 0.0 && cum > target) found = e0 + j;
            }
            found = __reduce_min_sync(0xffffffffu, found);
            my_last = __reduce_max_sync(0xffffffffu, my_last);
            if (lane == 0) out_tok[row] = found != 0x7fffffff ? found : max(my_last, 0);
        }
    }
    if (!ALONE) asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");       // no CTA leaves while its results may still be read
}

// ---------------------------------------------------------------------------------------------
// The whole call in one kernel, for calls whose rows are resident at once: a row is a cluster of C CTAs of
// 1024 threads, a CTA owns the slice [rank * S, rank * S + S) of the vocabulary in every vector.
//   stats     a warp per piece of a vector's slice, as in the stats pass; the CTAs' results are exchanged
//             through distributed shared memory and every CTA merges them and runs the accept tests itself
//   resample  a warp owns S / 32 neighbouring entries of position n, lanes side by side; their fp64
//             exponentials stay in registers; normalisers and masses are exchanged the same way, and the warp
//             whose stretch holds u2 * S walks it 32 entries at a time.
// These calls are bound by the chain of dependent steps, not by bytes: one row, k = 4, V = 32000 (1.15 MB)
// took 23.3 us as stats (36 busy warps), decide and resample kernels, 14.2 us as one (statistics 5, exchange and tests 3, resample 5).  Sums have a fixed order.
// ---------------------------------------------------------------------------------------------
constexpr int AR_THREADS = 1024, AR_WARPS = AR_THREADS / 32, AR_MAXC = 16;
constexpr int AR_TASKS = 2 * MAX_K + 1 + AR_WARPS;

__device__ __forceinline__ StatPartial cluster_read_stat(const StatPartial* local, uint32_t rank) {
    const uint32_t a = (uint32_t)__cvta_generic_to_shared(local);
    uint32_t r, w0, w1, w2, w3;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
    asm volatile("ld.shared::cluster.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(w0), "=r"(w1), "=r"(w2), "=r"(w3) : "r"(r) : "memory");
    StatPartial p;
    p.mx = __uint_as_float(w0); p.sum = __uint_as_float(w1); p.arg = (int)w2; p.pad = (int)w3;
    return p;
}
template <bool VEC, int PER>
__global__ void __launch_bounds__(AR_THREADS, 1)
accept_row_kernel(const float* __restrict__ tl, const float* __restrict__ dl, const int* __restrict__ onehot,
                  const int* tokens, int rows, int k, int V, float temperature, float lenience, uint64_t seed,
                  uint64_t step, int csize, int S, int pieces, int* __restrict__ n_acc, int* __restrict__ out_tok, int* seq,
                  int* status) {
    __shared__ StatPartial s_task[AR_TASKS];
    __shared__ StatPartial s_own[2 * MAX_K + 1];       // this CTA's slice of every vector
    __shared__ float s_mx[2 * MAX_K + 1], s_z[2 * MAX_K + 1];
    __shared__ int s_arg[2 * MAX_K + 1], s_acc[MAX_K + 1], s_point[MAX_K + 1], s_x[MAX_K + 1];
    __shared__ double s_u2[MAX_K + 1], s_ex[4], s_warp[AR_WARPS], s_warp2[AR_WARPS], s_tab[64];
    const int row = blockIdx.x / csize, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int rank = (int)cluster_rank();
    const bool greedy = temperature == 0.f;
    const float invT = greedy ? 1.f : 1.f / temperature;
    if (!greedy && tid < 64) s_tab[tid] = c_exp2_table[tid];
    pdl_wait();
    pdl_trigger();
    const int nvec = dl ? 2 * k + 1 : k + 1;
    const float* trow = tl + (long long)row * (k + 1) * V;
    const float* drow = dl ? dl + (long long)row * k * V : nullptr;
    // what the accept tests need besides the statistics travels while those are formed (thread i: position i)
    int x = 0;
    bool bad = false, point = true;
    float tx = 0.f, dx = 0.f;
    if (tid < k) {
        x = tokens[(long long)row * k + tid];
        bad = x < 0 || x >= V;
        point = !dl || (onehot && onehot[(long long)row * k + tid] != 0);
        if (!greedy && !bad) {
            tx = trow[(long long)tid * V + x];
            if (!point) dx = drow[(long long)tid * V + x];
        }
    }
    // ---- statistics of this CTA's slice
    const int lo = rank * S, hi = min(V, lo + S);
    const int plen = (S + pieces * 128 - 1) / (pieces * 128) * 128;
#pragma unroll 1
    for (int task = warp; task < nvec * pieces; task += AR_WARPS) {
        const int vec = task / pieces, from = lo + (task % pieces) * plen, to = min(hi, from + plen);
        const float* src = vec <= k ? trow + (long long)vec * V : drow + (long long)(vec - k - 1) * V;
        float mx = -INFINITY, sum = 0.f;
        int arg = 0x7fffffff;
#pragma unroll 1
        for (int e0 = from; e0 < to; e0 += ST_SUB) {
            float cur[32];
            load_sub<VEC>(src, e0, to, lane, cur);
            float bm = -INFINITY;
            int ba = 0x7fffffff;
#pragma unroll
            for (int j = 0; j < 32; ++j)
                if (cur[j] > bm) { bm = cur[j]; ba = sub_index<VEC>(e0, lane, j); }
            if (bm > mx) {
                sum = mx > -INFINITY ? sum * __expf((mx - bm) * invT) : 0.f;
                mx = bm; arg = ba;
            }
            if (!greedy && mx > -INFINITY) {
                float a = 0.f;
#pragma unroll
                for (int j = 0; j < 32; ++j) a += __expf((cur[j] - mx) * invT);
                sum += a;
            }
        }
        float wm = mx;
        int wa = arg;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const float om = __shfl_xor_sync(0xffffffffu, wm, o);
            const int oa = __shfl_xor_sync(0xffffffffu, wa, o);
            if (om > wm || (om == wm && oa < wa)) { wm = om; wa = oa; }
        }
        float scaled = (!greedy && mx > -INFINITY) ? sum * __expf((mx - wm) * invT) : 0.f;
        scaled = warp_sum(scaled);
        if (lane == 0) { StatPartial q; q.mx = wm; q.sum = scaled; q.arg = wa; q.pad = 0; s_task[task] = q; }
    }
    __syncthreads();
    if (tid < nvec) {
        float mx = -INFINITY, z = 0.f;
        int arg = 0x7fffffff;
        for (int c = 0; c < pieces; ++c) merge_stat(mx, z, arg, s_task[tid * pieces + c], invT);
        StatPartial q; q.mx = mx; q.sum = z; q.arg = arg; q.pad = 0;
        s_own[tid] = q;
    }
    cluster_sync_all();
    // (16 lanes a vector, one CTA's result each: a thread that walked the CTAs took 0.9 us longer)
#pragma unroll 1
    for (int i0 = 0; i0 < nvec; i0 += AR_THREADS / AR_MAXC) {
        const int i = i0 + tid / AR_MAXC, l = tid % AR_MAXC;
        StatPartial a;
        a.mx = -INFINITY; a.sum = 0.f; a.arg = 0x7fffffff; a.pad = 0;
        if (i < nvec && l < csize) a = cluster_read_stat(&s_own[i], (uint32_t)l);
        merge_stat_lanes<AR_MAXC>(a, invT);
        if (i < nvec && l == 0) { s_mx[i] = a.mx; s_z[i] = a.sum; s_arg[i] = a.arg; }
    }
    __syncthreads();
    // ---- the accept tests of all positions at once
    const double inv_temp = 1.0 / (double)temperature;
    if (tid <= k) {
        bool accept = false;
        double u2 = 0.0;
        if (greedy) {
            accept = tid < k && x == s_arg[tid];
        } else {
            const Philox4 r = philox4x32_10((uint32_t)tid, (uint32_t)row, (uint32_t)step, (uint32_t)(step >> 32), (uint32_t)seed,
                                            (uint32_t)(seed >> 32));
            u2 = word_uniform(r.w[1]);
            if (tid < k && !bad) accept = accept_test(word_uniform(r.w[0]), tx, s_mx[tid], s_z[tid], point, dx, point ? 0.f : s_mx[k + 1 + tid],
                                                      point ? 1.f : s_z[k + 1 + tid], inv_temp, lenience, s_tab);
        }
        if (tid < k && bad && rank == 0) set_status(status, CSD_ERR_BAD_TOKEN);
        s_acc[tid] = accept ? 1 : 0; s_point[tid] = point ? 1 : 0; s_x[tid] = bad ? 0 : x; s_u2[tid] = u2;
    }
    __syncthreads();
    int n = 0;
    while (n < k && s_acc[n]) ++n;
    if (rank == 0 && tid == 0) {
        if (greedy) {
            if (seq) seq[n] = s_arg[n];                // (`seq` may be `tokens`: every CTA has read those by now)
            out_tok[row] = s_arg[n];
        }
        n_acc[row] = n;
    }
    if (greedy) {
        cluster_sync_all();                            // no CTA leaves while another may still read its statistics
        return;
    }
    // ---- resample at position n
    const double max_t = (double)s_mx[n];
    int mode = n == k ? MODE_TARGET_ONLY : (s_point[n] ? MODE_RESID_POINT : MODE_RESID_LOGITS);
    const double max_q = mode == MODE_RESID_LOGITS ? (double)s_mx[k + 1 + n] : 0.0, u2 = s_u2[n];
    const int xn = s_x[n];
    const float* t = trow + (long long)n * V;
    const float* d = mode == MODE_RESID_LOGITS ? drow + (long long)n * V : nullptr;
    const int e0 = lo + warp * (PER * 32) + lane;      // entries e0 + 32 j
    double et[PER], ed[PER];
    {
        float tv[PER], dv[PER];
#pragma unroll
        for (int j = 0; j < PER; ++j) {
            const int e = e0 + 32 * j;
            tv[j] = e < hi ? t[e] : -INFINITY;
            dv[j] = d && e < hi ? d[e] : -INFINITY;
        }
#pragma unroll
        for (int j = 0; j < PER; ++j) {
            et[j] = exp_neg(((double)tv[j] - max_t) * inv_temp, s_tab);       // -inf (past the slice) gives 0
            ed[j] = d ? exp_neg(((double)dv[j] - max_q) * inv_temp, s_tab) : 0.0;
        }
    }
    double sp = 0.0, sq = 0.0;
#pragma unroll
    for (int j = 0; j < PER; ++j) { sp += et[j]; sq += ed[j]; }
    sp = warp_sum(sp); sq = warp_sum(sq);
    if (lane == 0) { s_warp[warp] = sp; s_warp2[warp] = sq; }
    __syncthreads();
    if (warp == 0) {
        sp = warp_sum(s_warp[lane]); sq = warp_sum(s_warp2[lane]);
        if (lane == 0) { s_ex[0] = sp; s_ex[1] = sq; }
    }
    cluster_sync_all();
    double Zp = 0.0, Zq = 0.0;
    {
        // (lanes 0-15 read the CTAs' Zp, lanes 16-31 their Zq)
        double a = lane % AR_MAXC < csize ? cluster_read_f64(&s_ex[lane / AR_MAXC], (uint32_t)(lane % AR_MAXC)) : 0.0;
#pragma unroll
        for (int o = AR_MAXC / 2; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
        Zp = __shfl_sync(0xffffffffu, a, 0); Zq = __shfl_sync(0xffffffffu, a, AR_MAXC);
    }
    auto resid = [&](int j) -> double {
        return e0 + 32 * j < hi ? residual_from(mode, et[j], ed[j], Zp, Zq, e0 + 32 * j == xn) : 0.0;
    };
    double mass_w = 0.0, run = 0.0, head = 0.0, total = 0.0;   // this warp's mass, the masses up to its end, before this CTA, all
    int owner = 0, forced = 0;
    double target = 0.0;
    // (a second time with the target law itself if the residual is empty)
#pragma unroll 1
    for (int pass = 0; pass < 2; ++pass) {
        double local = 0.0;
#pragma unroll
        for (int j = 0; j < PER; ++j) local += resid(j);
        mass_w = warp_sum(local);
        __syncthreads();
        if (lane == 0) s_warp[warp] = mass_w;
        __syncthreads();
        run = s_warp[lane];                            // inclusive prefix over the warps, lane = warp
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const double up = __shfl_up_sync(0xffffffffu, run, o);
            if (lane >= o) run += up;
        }
        if (tid == AR_THREADS - 1) s_ex[2 + pass] = run;
        cluster_sync_all();
        const double m = lane < csize ? cluster_read_f64(&s_ex[2 + pass], (uint32_t)lane) : 0.0;
        double incl = m;                               // inclusive prefix over the CTAs, lane = CTA
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const double up = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += up;
        }
        total = __shfl_sync(0xffffffffu, incl, csize - 1);
        if (pass == 0 && mode != MODE_TARGET_ONLY && (!(total > 0.0) || !isfinite(total))) { mode = MODE_TARGET_ONLY; continue; }
        // the CTA whose masses reach past u2 * total; rounding may leave none, then the last one that carries mass
        target = u2 * total;
        const unsigned past = __ballot_sync(0xffffffffu, lane < csize && incl > target);
        const unsigned some = __ballot_sync(0xffffffffu, m > 0.0);
        forced = past == 0;
        owner = past ? __ffs(past) - 1 : (some ? 31 - __clz(some) : 0);
        head = __shfl_sync(0xffffffffu, incl - m, rank);
        break;
    }
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");     // this CTA has read what it needs of the others
    if (rank == owner) {
        // ---- in it the warp (all lanes of all warps know the prefix), then the smallest index whose cumulative mass
        //      exceeds the target; forced, or where rounding leaves none: the last entry that carries mass
        const unsigned past = __ballot_sync(0xffffffffu, head + run > target);
        const unsigned some = __ballot_sync(0xffffffffu, s_warp[lane] > 0.0);
        const int wpick = past && !forced ? __ffs(past) - 1 : (some ? 31 - __clz(some) : 0);
        if (warp == wpick) {
            double cum = head + __shfl_sync(0xffffffffu, run, (wpick + 31) & 31) * (wpick > 0 ? 1.0 : 0.0);
            int pick = -1, last = -1;
#pragma unroll
            for (int j = 0; j < PER; ++j) {
                const double r = resid(j);
                double incl = r;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const double up = __shfl_up_sync(0xffffffffu, incl, o);
                    if (lane >= o) incl += up;
                }
                const unsigned hit = __ballot_sync(0xffffffffu, r > 0.0 && cum + incl > target);
                const unsigned mass = __ballot_sync(0xffffffffu, r > 0.0);
                const int first = lo + warp * (PER * 32) + 32 * j;
                if (pick < 0 && hit && !forced) pick = first + __ffs(hit) - 1;
                if (mass) last = first + 31 - __clz(mass);
                cum += __shfl_sync(0xffffffffu, incl, 31);
            }
            if (lane == 0) {
                const int y = pick >= 0 ? pick : max(last, 0);
                if (seq) seq[n] = y;
                out_tok[row] = y;
            }
        }
    }
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");       // no CTA leaves while its results may still be read
}

// The layout for `room` bytes of scratch: chunks of 1024 logits for the resample where that holds them, else of 4096.  (V = 128256: 64
// rows, k = 4 92 / 104 us a call, k = 16 214 / 223; 320 rows, k = 1 196 / 207.)
static csd_status accept_layout_in(int rows, int k, int V, size_t room, AcceptLayout& L) {
    const AcceptLayout least = accept_layout(rows, k, V, 4);
    if (room < least.total) return CSD_ERR_CAPACITY;
    if (least.pieces > 65535) return CSD_ERR_UNSUPPORTED;
    L = accept_layout(rows, k, V);
    if (room < L.total || L.pieces > 65535) L = least;
    return CSD_OK;
}

static int accept_sm_count() {
    static int n = 0;
    if (n == 0) {
        int dev = 0;
        if (cudaGetDevice(&dev) != cudaSuccess ||
            cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0)
            n = 148;
    }
    return n;
}

// The table of 2^(j/64), correctly rounded, goes to constant memory once per device.
static csd_status exp_table_ready() {
    static bool done[MAX_DEVICES];
    static std::mutex mu;
    int dev = 0;
    CSD_CUDA(cudaGetDevice(&dev));
    if (dev < 0 || dev >= MAX_DEVICES) return CSD_ERR_UNSUPPORTED;
    std::lock_guard<std::mutex> lk(mu);
    if (!done[dev]) {
        double tab[64];
        for (int j = 0; j < 64; ++j) tab[j] = exp2((double)j / 64.0);
        CSD_CUDA(cudaMemcpyToSymbol(c_exp2_table, tab, sizeof(tab)));
        done[dev] = true;
    }
    return CSD_OK;
}

// Whether clusters of `csize` CTAs of the fused resample kernel can run on the current device.
static bool fused_resample_ok(int csize) {
    static PerDevice known[RF_MAXC + 1];
    if (csize < 1 || csize > RF_MAXC) return false;
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess) { (void)cudaGetLastError(); return false; }
    return known[csize].get(dev, [csize] {
        cudaLaunchConfig_t cfg = cudaLaunchConfig_t{};
        cudaLaunchAttribute attr[1];
        cfg.gridDim = dim3((unsigned)csize); cfg.blockDim = dim3(RF_THREADS);
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = (unsigned)csize; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr; cfg.numAttrs = 1;
        int n = 0;
        const bool ok = cudaOccupancyMaxActiveClusters(&n, csize == 1 ? resample_fused_kernel<true> : resample_fused_kernel<false>, &cfg) == cudaSuccess && n >= 1;
        if (!ok) (void)cudaGetLastError();
        return ok ? 1 : 0;
    }) == 1;
}

// Clusters of `csize` CTAs of the one-kernel form that are resident at once on the current device (0: none).  The opt-in to
// clusters above 8 is an attribute of the kernel on one device, so both are settled for each device.
template <bool VEC, int PER>
static int row_clusters(int csize) {
    static PerDevice known[AR_MAXC + 1];
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess) { (void)cudaGetLastError(); return 0; }
    return known[csize].get(dev, [csize] {
        int n = 0;
        bool ok = true;
        if (csize > 8)
            ok = cudaFuncSetAttribute(accept_row_kernel<VEC, PER>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess;
        if (ok) {
            cudaLaunchConfig_t cfg = cudaLaunchConfig_t{};
            cudaLaunchAttribute attr[1];
            cfg.gridDim = dim3((unsigned)csize); cfg.blockDim = dim3(AR_THREADS);
            attr[0].id = cudaLaunchAttributeClusterDimension;
            attr[0].val.clusterDim.x = (unsigned)csize; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
            cfg.attrs = attr; cfg.numAttrs = 1;
            ok = cudaOccupancyMaxActiveClusters(&n, accept_row_kernel<VEC, PER>, &cfg) == cudaSuccess;
        }
        if (!ok) { (void)cudaGetLastError(); n = 0; }
        return n;
    });
}

template <bool VEC, int PER>
static csd_status launch_accept_row(const float* tl, const float* dl, const int* onehot, const int* tokens, int rows, int k,
                                    int V, float temperature, float lenience, uint64_t seed, uint64_t step, int csize,
                                    int* n_acc, int* out_tok, int* seq, int* status, cudaStream_t st, bool* done) {
    *done = false;
    const int S = ((V + csize - 1) / csize + 3) & ~3, nvec = dl ? 2 * k + 1 : k + 1;
    // (a CTA takes in about 40 GB/s here: beyond about 320 KB of slices the stats pass over all SMs is faster; one row,
    // V = 128256: k = 4, 289 KB, 29.6 us against 34.3; k = 8, 545 KB, 35.0 against 34.3)
    if ((long long)nvec * S * 4 > 320 * 1024 || row_clusters<VEC, PER>(csize) < rows) return CSD_OK;
    // pieces of a vector's slice, of at least 1024 logits: enough for every warp, fewer where that saves batches of the busiest warp (2 rows,
    // k 6, V 50000, 13 vectors: 39 tasks for 32 warps 19.7 us, 26 of them 17.8)
    auto batches = [&](int n) {
        const int plen = (S + n * 128 - 1) / (n * 128) * 128;
        return (nvec * n + AR_WARPS - 1) / AR_WARPS * ((plen + ST_SUB - 1) / ST_SUB);
    };
    int pieces = (AR_WARPS + nvec - 1) / nvec;
    if (pieces > (S + ST_SUB - 1) / ST_SUB) pieces = (S + ST_SUB - 1) / ST_SUB;
    for (int n = pieces - 1; n >= 1; --n)
        if (batches(n) < batches(pieces)) pieces = n;
    cudaLaunchConfig_t cfg = cudaLaunchConfig_t{};
    cudaLaunchAttribute attr[2];
    cfg.gridDim = dim3((unsigned)(rows * csize)); cfg.blockDim = dim3(AR_THREADS); cfg.dynamicSmemBytes = 0; cfg.stream = st;
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)csize; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr; cfg.numAttrs = 2;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, accept_row_kernel<VEC, PER>, tl, dl, onehot, tokens, rows, k, V, temperature,
                                             lenience, seed, step, csize, S, pieces, n_acc, out_tok, seq, status);
    if (e == cudaErrorInvalidConfiguration || e == cudaErrorInvalidClusterSize || e == cudaErrorLaunchOutOfResources) {
        (void)cudaGetLastError();                        // a configuration the device does not take: left to the passes
        return CSD_OK;
    }
    CSD_CUDA(e);
    count_launch();
    *done = true;
    return CSD_OK;
}

// The three passes on scratch `ws` (accept_layout bytes).  Every word a pass reads is written by an
// earlier pass of the same call (the decide pass clears the resample tickets), so the scratch
// needs no initialisation.
static csd_status run_accept(const float* tl, const float* dl_in, const int32_t* onehot, const int32_t* tokens, int rows,
                             int k, int V, float temperature, float lenience, uint64_t seed, uint64_t step,
                             int32_t* n_acc, int32_t* out_tok, char* ws, const AcceptLayout& L, int* status,
                             cudaStream_t st, int32_t* seq = nullptr, bool* seq_written = nullptr) {
    StatPartial* part = (StatPartial*)(ws + L.part_off);
    RowInfo* info = (RowInfo*)(ws + L.info_off);
    unsigned* tickets = (unsigned*)(ws + L.ticket_off);
    const bool greedy = temperature == 0.f;
    const float invT = greedy ? 1.f : 1.f / temperature;
    const bool use_d = dl_in != nullptr && k > 0 && !greedy;
    const float* dl = use_d ? dl_in : nullptr;
    const long long n_tvec = (long long)rows * (k + 1);
    const long long nvec = n_tvec + (use_d ? (long long)rows * k : 0);
    if (nvec > 0x7fffffffLL) return CSD_ERR_UNSUPPORTED;
    const bool vec_ok = (V % 4 == 0) && (((uintptr_t)tl & 15) == 0) && (!use_d || ((uintptr_t)dl & 15) == 0);
    // One kernel while its clusters are all resident; smallest power of two that leaves a CTA at most
    // 4096 entries and 320 KB, doubled while that leaves it 512 and the rows still fit, halved while it takes that for all
    // rows to be resident (k 4, V 32000: 16 rows 24.4 -> 23.1 us, 30 rows 29.5 -> 23.9; in two waves of clusters of 8 27.4 and 30.7).
    if (!greedy) {
        const csd_status ts = exp_table_ready();
        if (ts != CSD_OK) return ts;
    }
    if (V <= AR_MAXC * 8192) {
        int csize = 1;
        while (csize < 8 && (V + csize - 1) / csize > 4096) csize *= 2;
        // (clusters of 16: 2 rows, k 6, V 50000 24.0 -> 17.8 us, 1 row, k 4, V 64000 22.0 -> 17.8, k 16, V 32000 23.3 -> 21.2; k 4, V 32000 13.6 -> 14.2)
        if (V > 8 * 4096 || (csize == 8 && (long long)(use_d ? 2 * k + 1 : k + 1) * V / 8 * 4 > 320 * 1024)) csize = 16;
        while (csize < 8 && rows * csize * 2 <= accept_sm_count() && V / (csize * 2) >= 512) csize *= 2;
        bool done = false;
        csd_status s = CSD_OK;
        for (;; csize /= 2) {
            const int S = ((V + csize - 1) / csize + 3) / 4 * 4;
            if (S > 8192) break;
            if (vec_ok)
                s = S > 4096 ? launch_accept_row<true, 8>(tl, dl, onehot, tokens, rows, k, V, temperature, lenience, seed, step, csize, n_acc, out_tok, seq, status, st, &done)
                             : launch_accept_row<true, 4>(tl, dl, onehot, tokens, rows, k, V, temperature, lenience, seed, step, csize, n_acc, out_tok, seq, status, st, &done);
            else
                s = S > 4096 ? launch_accept_row<false, 8>(tl, dl, onehot, tokens, rows, k, V, temperature, lenience, seed, step, csize, n_acc, out_tok, seq, status, st, &done)
                             : launch_accept_row<false, 4>(tl, dl, onehot, tokens, rows, k, V, temperature, lenience, seed, step, csize, n_acc, out_tok, seq, status, st, &done);
            if (s != CSD_OK || done || csize == 1) break;
        }
        if (seq_written) *seq_written = done && seq;
        if (s != CSD_OK || done) return s;
    }
    const long long items = nvec * L.nchunk_a;
    long long ctas = (items + ST_THREADS / 32 - 1) / (ST_THREADS / 32);
    const long long cap = (long long)accept_sm_count() * 2;       // two resident CTAs per SM, grid-stride beyond
    if (ctas > cap) ctas = cap;
    // both launched with programmatic stream serialisation: they are resident and waiting when their
    // predecessor retires (in the cascade that is the output head of the review forward)
    {
        PdlLaunch ls(dim3((unsigned)ctas), dim3(ST_THREADS), 0, st);
        const int greedy_i = greedy ? 1 : 0;
        if (vec_ok)
            CSD_CUDA(cudaLaunchKernelEx(&ls.cfg, accept_stats_kernel<true>, tl, dl, n_tvec, V, invT, greedy_i, part, L.nchunk_a, items));
        else
            CSD_CUDA(cudaLaunchKernelEx(&ls.cfg, accept_stats_kernel<false>, tl, dl, n_tvec, V, invT, greedy_i, part, L.nchunk_a, items));
        PdlLaunch ld(dim3((unsigned)rows), dim3(DC_THREADS), 0, st);
        CSD_CUDA(cudaLaunchKernelEx(&ld.cfg, accept_decide_kernel, tl, dl, (const int*)onehot, (const int*)tokens, rows, k, V,
                                    temperature, lenience, seed, step, (const StatPartial*)part, L.nchunk_a, (int*)n_acc,
                                    (int*)out_tok, info, tickets, status));
    }
    count_launch(2);
    const int csize = (V + RF_SLICE - 1) / RF_SLICE;
    // A row that fits one cluster goes to the fused kernel.  Measured, fused / passes: 10 rows, k 8, V 50000 29.7 / 31.4 us a call, 20 rows 44.9
    // / 39.5; 64 rows, k 16, V 32000 77.9 / 71.7, k 4 43.0 / 37.4; 64 rows, k 4, V 60000 75.9 / 54.5: since the passes end in a kernel
    // of their own, the line lies too high.
    if (!greedy && fused_resample_ok(csize)) {
        cudaLaunchConfig_t cfg = cudaLaunchConfig_t{};
        cudaLaunchAttribute attr[2];
        cfg.gridDim = dim3((unsigned)(rows * csize)); cfg.blockDim = dim3(RF_THREADS); cfg.dynamicSmemBytes = 0; cfg.stream = st;
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = (unsigned)csize; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
        attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[1].val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = attr; cfg.numAttrs = 2;
        CSD_CUDA(cudaLaunchKernelEx(&cfg, csize == 1 ? resample_fused_kernel<true> : resample_fused_kernel<false>, tl, dl, k, V, temperature, (const RowInfo*)info, csize,
                                    (int*)out_tok));
        count_launch();
    } else if (!greedy) {
        const int nch = L.chunks;
        ChunkSums* sums = (ChunkSums*)(ws + L.sums_off);
        unsigned short* lists = (unsigned short*)(ws + L.lists_off);
        // warps a block: fewer while that leaves SMs without one (2 rows, k 15, V 128256 31.8 -> 29.2 us, 4 rows, k 16 34.8 -> 34.1)
        int warps = RS_THREADS / 32;
        while (warps > 1 && (long long)rows * nch < (long long)warps * accept_sm_count()) warps /= 2;
        PdlLaunch lo(dim3((unsigned)(((long long)rows * nch + warps - 1) / warps)), dim3((unsigned)warps * 32), 0, st);
        CSD_CUDA(cudaLaunchKernelEx(&lo.cfg, resample_sums_kernel, tl, dl, rows, k, V, temperature, (const RowInfo*)info, sums, lists, nch,
                                    L.sets));
        // CTAs a row, for chunks that are formed anew: as many as fit at once, at least a chunk a warp.  (A chunk a warp at any number
        // of rows: 64 rows of laws that nearly agree 106 -> 102 us, others, whose further CTAs leave at once, 217 -> 220.)
        int per_row = (nch + RS_THREADS / 32 - 1) / (RS_THREADS / 32);
        if ((long long)per_row * rows > 3 * accept_sm_count()) per_row = max(1, 3 * accept_sm_count() / rows);
        PdlLaunch lp(dim3((unsigned)(rows * per_row)), dim3(RS_THREADS), 0, st);
        CSD_CUDA(cudaLaunchKernelEx(&lp.cfg, resample_pick_kernel, tl, dl, k, V, temperature, (const RowInfo*)info, sums, (const unsigned short*)lists,
                                    tickets, nch, L.sets, per_row, (int*)out_tok));
        count_launch(2);
    }
    CSD_CUDA(cudaGetLastError());
    return CSD_OK;
}

}  // namespace csd

using namespace csd;

extern "C" size_t csd_spec_accept_workspace_bytes(int rows, int k, int V) {
    if (rows < 0 || k < 0 || V < 1) return 0;
    return accept_layout(rows, k, V).total;
}

namespace csd {
csd_status accept_into(const float* target_logits_dev, const float* draft_logits_dev, const int32_t* onehot_dev,
                       const int32_t* draft_tokens_dev, int rows, int k, int V, float temperature, float lenience, uint64_t seed,
                       uint64_t step, int32_t* n_accepted_dev, int32_t* out_token_dev, void* workspace_dev,
                       size_t workspace_bytes, void* stream, int32_t* seq, bool* seq_written) {
    if (rows < 0 || k < 0 || k > MAX_K || V < 1 || !(temperature >= 0.f) || !(lenience >= 1.f))
        return CSD_ERR_INVALID_ARG;
    if (rows == 0) return CSD_OK;
    if (!target_logits_dev || !n_accepted_dev || !out_token_dev || !workspace_dev) return CSD_ERR_INVALID_ARG;
    if (k > 0 && !draft_tokens_dev) return CSD_ERR_INVALID_ARG;
    if (((uintptr_t)workspace_dev & 255) != 0) return CSD_ERR_INVALID_ARG;
    AcceptLayout L;
    const csd_status fits = accept_layout_in(rows, k, V, workspace_bytes, L);
    if (fits != CSD_OK) return fits;
    int* status = status_word_device();
    if (!status) return CSD_ERR_CUDA;
    return run_accept(target_logits_dev, draft_logits_dev, onehot_dev, draft_tokens_dev, rows, k, V, temperature, lenience,
                      seed, step, n_accepted_dev, out_token_dev, (char*)workspace_dev, L, status, (cudaStream_t)stream, seq,
                      seq_written);
}
}  // namespace csd

extern "C" csd_status csd_spec_accept(const float* target_logits_dev, const float* draft_logits_dev,
                                      const int32_t* onehot_dev, const int32_t* draft_tokens_dev, int rows, int k,
                                      int V, float temperature, float lenience, uint64_t seed, uint64_t step,
                                      int32_t* n_accepted_dev, int32_t* out_token_dev, void* workspace_dev,
                                      size_t workspace_bytes, void* stream) {
    return accept_into(target_logits_dev, draft_logits_dev, onehot_dev, draft_tokens_dev, rows, k, V, temperature, lenience, seed,
                       step, n_accepted_dev, out_token_dev, workspace_dev, workspace_bytes, stream, nullptr, nullptr);
}


// ---------------------------------------------------------------------------------------------
// Greedy acceptance along a tree of drafted tokens (tree attention, Section 5.1 / Appendix B).
// ---------------------------------------------------------------------------------------------
namespace csd {

struct TreeShape { int parent[CSD_MAX_ROWS]; };

// arg-max of every row of the target logits (smallest index on ties), one CTA per row
__global__ void __launch_bounds__(256)
tree_argmax_kernel(const float* __restrict__ logits, int V, int* __restrict__ arg) {
    pdl_wait();
    pdl_trigger();
    const float* x = logits + (size_t)blockIdx.x * V;
    float best = -INFINITY;
    int at = 0x7fffffff;
    for (int i = threadIdx.x; i < V; i += 256) {
        const float v = x[i];
        if (v > best || at == 0x7fffffff) { best = v; at = i; }
    }
    __shared__ float s_v[256];
    __shared__ int s_i[256];
    s_v[threadIdx.x] = best; s_i[threadIdx.x] = at;
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
        if (threadIdx.x < o) {
            const float ov = s_v[threadIdx.x + o];
            const int oi = s_i[threadIdx.x + o];
            if (ov > s_v[threadIdx.x] || (ov == s_v[threadIdx.x] && oi < s_i[threadIdx.x])) { s_v[threadIdx.x] = ov; s_i[threadIdx.x] = oi; }
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) arg[blockIdx.x] = s_i[0] == 0x7fffffff ? 0 : s_i[0];
}

// out[0] = tokens emitted, out[1] = leading rows of the accepted path that are a chain 0, 1, 2, ..
// (their cache entries are valid), out[2 ..] = the emitted tokens, out[2 + m ..] = rows of the path
__global__ void tree_walk_kernel(const int* __restrict__ arg, const int* __restrict__ tokens, const TreeShape shape, int m,
                                 int V, int* __restrict__ out, int* status) {
    if (threadIdx.x != 0) return;
    int cur = 0, n_out = 0, n_valid = 1;
    bool chain = true;
    out[2 + m] = 0;
    while (true) {
        const int y = arg[cur];
        out[2 + n_out] = y;
        ++n_out;
        int nxt = -1;
        for (int c = cur + 1; c < m; ++c) {
            const int t = tokens[c];
            if (t < 0 || t >= V) { set_status(status, CSD_ERR_BAD_TOKEN); continue; }
            if (shape.parent[c] == cur && t == y) { nxt = c; break; }
        }
        if (nxt < 0 || n_out >= m) break;
        out[2 + m + n_out] = nxt;
        chain = chain && nxt == n_out;
        if (chain) n_valid = n_out + 1;
        cur = nxt;
    }
    out[0] = n_out;
    out[1] = n_valid;
}

}  // namespace csd

extern "C" csd_status csd_tree_accept_greedy(const float* target_logits_dev, const int32_t* tokens_dev,
                                             const int32_t* parent_host, int n_rows, int V, int32_t* out_dev, void* stream) {
    if (!target_logits_dev || !tokens_dev || !parent_host || !out_dev || n_rows < 1 || n_rows > CSD_MAX_ROWS || V < 1)
        return CSD_ERR_INVALID_ARG;
    TreeShape shape;
    for (int r = 0; r < CSD_MAX_ROWS; ++r) shape.parent[r] = -2;
    for (int r = 0; r < n_rows; ++r) {
        const int p = parent_host[r];
        if (r == 0 ? p != -1 : (p < 0 || p >= r)) return CSD_ERR_INVALID_ARG;
        shape.parent[r] = p;
    }
    int* status = status_word_device();
    if (!status) return CSD_ERR_CUDA;
    cudaStream_t st = (cudaStream_t)stream;
    int* arg = (int*)out_dev + 2 + 2 * n_rows;
    PdlLaunch la(dim3((unsigned)n_rows), dim3(256), 0, st);
    CSD_CUDA(cudaLaunchKernelEx(&la.cfg, tree_argmax_kernel, target_logits_dev, V, arg));
    tree_walk_kernel<<<1, 32, 0, st>>>((const int*)arg, (const int*)tokens_dev, shape, n_rows, V, (int*)out_dev, status);
    count_launch(2);
    CSD_CUDA(cudaGetLastError());
    return CSD_OK;
}

// ---------------------------------------------------------------------------------------------
// Variant for callers that must not allocate: its scratch is a fixed array inside the library.
// ---------------------------------------------------------------------------------------------
namespace csd {
constexpr size_t STATIC_SCRATCH_BYTES = (size_t)2 << 20;   // 2 MiB, held by every GPU that loads the library
static __device__ __align__(256) unsigned char g_accept_scratch[STATIC_SCRATCH_BYTES];
static void* g_accept_scratch_ptr[MAX_DEVICES];             // device address of the array, per device
static std::mutex g_accept_scratch_mu;
}  // namespace csd

extern "C" size_t csd_spec_accept_static_capacity(void) { return STATIC_SCRATCH_BYTES; }

extern "C" csd_status csd_spec_accept_static(const float* target_logits_dev, const float* draft_logits_dev,
                                             const int32_t* onehot_dev, const int32_t* draft_tokens_dev, int rows,
                                             int k, int V, float temperature, float lenience, uint64_t seed,
                                             uint64_t step, int32_t* n_accepted_dev, int32_t* out_token_dev,
                                             void* stream) {
    if (rows < 0 || k < 0 || k > MAX_K || V < 1 || !(temperature >= 0.f) || !(lenience >= 1.f))
        return CSD_ERR_INVALID_ARG;
    if (rows == 0) return CSD_OK;
    if (!target_logits_dev || !n_accepted_dev || !out_token_dev) return CSD_ERR_INVALID_ARG;
    if (k > 0 && !draft_tokens_dev) return CSD_ERR_INVALID_ARG;
    AcceptLayout L;
    const csd_status fits = accept_layout_in(rows, k, V, STATIC_SCRATCH_BYTES, L);
    if (fits != CSD_OK) return fits;
    // Set-up, once per device: in host code the array's name is only a handle, so ask the runtime
    // for the address the kernels can use.  Nothing is allocated here.
    int dev = 0;
    CSD_CUDA(cudaGetDevice(&dev));
    if (dev < 0 || dev >= MAX_DEVICES) return CSD_ERR_UNSUPPORTED;
    char* ws = nullptr;
    {
        std::lock_guard<std::mutex> lk(g_accept_scratch_mu);
        if (!g_accept_scratch_ptr[dev]) {
            void* p = nullptr;
            CSD_CUDA(cudaGetSymbolAddress(&p, g_accept_scratch));
            g_accept_scratch_ptr[dev] = p;
        }
        ws = (char*)g_accept_scratch_ptr[dev];
    }
    // (bad token ids are not recorded in the status word here: looking that word up may allocate)
    return run_accept(target_logits_dev, draft_logits_dev, onehot_dev, draft_tokens_dev, rows, k, V, temperature, lenience,
                      seed, step, n_accepted_dev, out_token_dev, ws, L, nullptr, (cudaStream_t)stream);
}
