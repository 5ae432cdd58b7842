// Where the passes of the accept call keep what they hand on, in the caller's scratch.  Host code only.
#pragma once
#include <cstddef>

namespace csd {

constexpr int ST_CHUNK = 8192;   // logits per warp item of the stats pass
constexpr int RS_CHUNK = 512;    // logits of a set: 8 neighbours a lane, twice
constexpr int RS_SETS = 2;       // sets of a chunk of the resample passes (times 4 where the scratch is small)
constexpr int RS_LIST = 6;       // undecided entries a chunk can list

struct alignas(16) StatPartial {
    float mx;
    float sum;   // sum exp((x - mx) * invT) over the piece
    int arg;     // smallest index attaining mx
    int pad;
};

struct alignas(16) RowInfo {
    int n;        // first rejected position (k if none)
    int mode;
    int x;        // drafted token at position n (point-mass / validation)
    int pad;
    double max_t; // max target logit at position n
    double max_q; // max draft logit at position n
    double u2;    // resampling uniform
    float z_t, z_q;   // sums of the exponentials at position n as the stats pass has them (fp32)
};

struct ChunkSums { double p, q, a, b; };   // all entries' exponentials of both laws; those of the entries that stay; later b: the mass

struct AcceptLayout {
    size_t part_off, info_off, sums_off, lists_off, ticket_off, total;
    int nchunk_a, pieces, chunks, sets;    // pieces of the stats pass; of 512 * times logits; chunks of the resample, of `sets` sets
};

// times: 1, or 4 where the scratch is small
inline AcceptLayout accept_layout(int rows, int k, int V, int times = 1) {
    auto up = [](size_t n) { return (n + 255) / 256 * 256; };
    AcceptLayout L;
    L.nchunk_a = (V + ST_CHUNK - 1) / ST_CHUNK;
    L.pieces = (int)(((long long)V + times * RS_CHUNK - 1) / (times * RS_CHUNK));
    L.chunks = (L.pieces + RS_SETS - 1) / RS_SETS;
    L.sets = times * RS_SETS;
    const size_t r = (size_t)rows, vectors = r * (2 * (size_t)k + 1);
    L.part_off = 0;
    L.info_off = up(vectors * L.nchunk_a * sizeof(StatPartial));
    L.sums_off = L.info_off + up(r * sizeof(RowInfo));
    L.lists_off = L.sums_off + r * L.chunks * sizeof(ChunkSums);
    L.ticket_off = L.lists_off + r * L.chunks * RS_LIST * sizeof(unsigned short);
    // What callers have been asked for all along: 24 bytes a piece and 24 a row, in four parts on 256-byte boundaries.  A chunk's 44
    // bytes and a row's ticket fit for any number of pieces: n of them give 24 n + 24, n / 2 chunks rounded up take at most 22 n + 26.
    static_assert(RS_SETS == 2 && sizeof(ChunkSums) + RS_LIST * sizeof(unsigned short) == 44, "room of a chunk");
    L.total = L.sums_off + up(r * L.pieces * 16) + up(r * L.pieces * 8) + up(r * 16) + up(r * 8);
    return L;
}

}  // namespace csd
