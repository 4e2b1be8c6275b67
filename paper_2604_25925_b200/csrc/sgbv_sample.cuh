// Inverse-CDF sampling over a vocabulary row by one CTA: the pieces shared by the finishing kernels
// (Eq. 4's residual draw, the bonus draw from the target row, Algorithm 2's draw, K-SEQ's residual).
// Summation order is fixed (ascending vocabulary index, float64 running sums), so draws are reproducible.
#pragma once

#include <limits.h>

#include "sgbv_cluster.cuh"
#include "sgbv_common.cuh"

namespace sgbv {

constexpr int kSampleMaxWarps = 32;  // CTAs of up to 1024 threads
constexpr int kEpt = 1;              // elements per thread inside one tile (threads beyond the tile hold none)

// Shared-memory scratch of the routines below (one per CTA).
struct SampleScratch {
    double warp[kSampleMaxWarps];
    int pick[2];
    int i[4];
    double d[2];
};

struct Pick {
    int first;  // smallest index whose cumulative weight exceeds the target, INT_MAX if none
    int last;   // largest index with positive weight, -1 if none
};

// Inverse CDF inside one tile: element x0 + kEpt*tid + j has weight wfun(x). base = cumulative
// weight before the tile. All threads must call.
template <typename F>
__device__ Pick pick_in_tile(int x0, int x1, double base, double target, F wfun, double *sh_warp, int *sh_pick) {
    const int tid = threadIdx.x, lane = tid & 31, wid = warp_index();
    float w[kEpt];
    double local = 0.0;
#pragma unroll
    for (int j = 0; j < kEpt; ++j) {
        const int x = x0 + kEpt * tid + j;
        w[j] = (x < x1) ? wfun(x) : 0.0f;
        local += (double)w[j];
    }
    double incl = local;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        double v = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += v;
    }
    if (tid == 0) {
        sh_pick[0] = INT_MAX;
        sh_pick[1] = -1;
    }
    if (lane == 31) sh_warp[wid] = incl;
    __syncthreads();
    // mass of the warps before this one: a butterfly over the lanes instead of a loop over the warps
    const double wv = lane < (int)(blockDim.x >> 5) ? sh_warp[lane] : 0.0;
    const double off = base + warp_sum(lane < wid ? wv : 0.0);
    double cum = off + incl - local;
    int first = INT_MAX, last = -1;
#pragma unroll
    for (int j = 0; j < kEpt; ++j) {
        cum += (double)w[j];
        const int x = x0 + kEpt * tid + j;
        if (w[j] > 0.0f) {
            last = x;
            if (cum > target) first = min(first, x);
        }
    }
    // (one atomic per warp: one per thread, on two words, took a thousand cycles)
    first = __reduce_min_sync(0xffffffffu, first);
    last = __reduce_max_sync(0xffffffffu, last);
    if (lane == 0) {
        if (last >= 0) atomicMax(&sh_pick[1], last);
        if (first != INT_MAX) atomicMin(&sh_pick[0], first);
    }
    __syncthreads();
    Pick p{sh_pick[0], sh_pick[1]};
    __syncthreads();
    return p;
}

// First tile whose inclusive prefix of the tile sums exceeds the target (float64, ascending
// vocabulary order), found by the whole block: every thread owns a contiguous run of tiles, the
// runs' totals are scanned across the block, and each thread searches its own run.  If rounding
// leaves no such tile, the last tile with positive mass is taken, with a base that makes the
// in-tile search fall back to its last positive element.  scale[t] (may be NULL) multiplies tile
// t's sum.  relative: `target` is a fraction of the total of all tile sums (computed here on the
// way) instead of a mass.  All threads must call.  Results: sh_i[2] = tile, sh_d[0] = mass before it,
// sh_d[1] = target.
static __device__ void locate_tile(const float *partials, const float *scale, int ntiles, double target, bool relative,
                            int *sh_i, double *sh_d, double *sh_warp) {
    const int tid = threadIdx.x, lane = tid & 31, wid = warp_index();
    const int nthreads = blockDim.x;
    const int per = (ntiles + nthreads - 1) / nthreads;
    const int t0 = min(ntiles, tid * per), t1 = min(ntiles, t0 + per);
    // the thread's tile sums: the first four stay in registers for the search below
    constexpr int kKeep = 4;
    double kept[kKeep];
    double local = 0.0;
#pragma unroll
    for (int e = 0; e < kKeep; ++e) {
        const int t = t0 + e;
        kept[e] = (t < t1) ? (double)partials[t] * (scale ? (double)scale[t] : 1.0) : 0.0;
        local += kept[e];
    }
    for (int t = t0 + kKeep; t < t1; ++t) local += (double)partials[t] * (scale ? (double)scale[t] : 1.0);
    double incl = local;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const double v = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += v;
    }
    if (tid == 0) {
        sh_i[2] = INT_MAX;  // first tile that crosses the target
        sh_i[3] = -1;       // last tile with positive mass
    }
    if (lane == 31) sh_warp[wid] = incl;
    __syncthreads();
    // the warps' totals: every warp adds up those of the warps before it (and all of them) with a butterfly
    // over its lanes instead of one after the other
    const double wv = lane < (nthreads >> 5) ? sh_warp[lane] : 0.0;
    const double cum0 = incl - local + warp_sum(lane < wid ? wv : 0.0);
    if (relative) target *= warp_sum(wv);  // the target is given as a fraction of the total of all tiles
    double cum = cum0;
    int first = INT_MAX, lastpos = -1;
    double base = 0.0;
    for (int t = t0; t < t1; ++t) {
        double v;
        if (t - t0 < kKeep) {
            v = kept[0];
#pragma unroll
            for (int e = 1; e < kKeep; ++e)
                if (t - t0 == e) v = kept[e];
        } else {
            v = (double)partials[t] * (scale ? (double)scale[t] : 1.0);
        }
        if (v > 0.0) lastpos = t;
        if (first == INT_MAX && cum + v > target) {
            first = t;
            base = cum;
        }
        cum += v;
    }
    const int first_w = __reduce_min_sync(0xffffffffu, first), last_w = __reduce_max_sync(0xffffffffu, lastpos);
    if (lane == 0) {
        if (first_w != INT_MAX) atomicMin(&sh_i[2], first_w);
        if (last_w >= 0) atomicMax(&sh_i[3], last_w);
    }
    __syncthreads();
    if (first != INT_MAX && sh_i[2] == first) sh_d[0] = base;  // exactly one thread owns that tile
    __syncthreads();
    if (tid == 0) {
        if (sh_i[2] == INT_MAX) {
            sh_i[2] = max(sh_i[3], 0);
            sh_d[0] = -INFINITY;
        }
        sh_d[1] = target;
    }
    __syncthreads();
}

// The 8 entries of a 256-entry tile that one lane takes when the row can be read in 16-byte pieces (the row starts
// on a 16-byte boundary and V is a multiple of the entries per piece, so a piece lies inside the row or past it).
template <typename T>
__device__ __forceinline__ void load_tile_pieces(const T *zq, int tile, bool in, int V, int lane, float (&z)[kTile / 32]);
template <>
__device__ __forceinline__ void load_tile_pieces<float>(const float *zq, int tile, bool in, int V, int lane,
                                                        float (&z)[kTile / 32]) {
    const float ninf = -INFINITY;
    const int xa = tile * kTile + lane * 4, xb = xa + kTile / 2;
    const float4 a = (in && xa < V) ? __ldg(reinterpret_cast<const float4 *>(zq + xa)) : make_float4(ninf, ninf, ninf, ninf);
    const float4 b = (in && xb < V) ? __ldg(reinterpret_cast<const float4 *>(zq + xb)) : make_float4(ninf, ninf, ninf, ninf);
    z[0] = a.x; z[1] = a.y; z[2] = a.z; z[3] = a.w;
    z[4] = b.x; z[5] = b.y; z[6] = b.z; z[7] = b.w;
}
template <>
__device__ __forceinline__ void load_tile_pieces<uint16_t>(const uint16_t *zq, int tile, bool in, int V, int lane,
                                                           float (&z)[kTile / 32]) {
    const uint32_t ninf2 = 0xff80ff80u;  // two bf16 -inf
    const int xa = tile * kTile + lane * 8;
    const uint4 a = (in && xa < V) ? __ldg(reinterpret_cast<const uint4 *>(zq + xa)) : make_uint4(ninf2, ninf2, ninf2, ninf2);
    z[0] = __uint_as_float(a.x << 16); z[1] = __uint_as_float(a.x & 0xffff0000u);
    z[2] = __uint_as_float(a.y << 16); z[3] = __uint_as_float(a.y & 0xffff0000u);
    z[4] = __uint_as_float(a.z << 16); z[5] = __uint_as_float(a.z & 0xffff0000u);
    z[6] = __uint_as_float(a.w << 16); z[7] = __uint_as_float(a.w & 0xffff0000u);
}


// Statistics of tiles t0..t1-1 of a row, by the whole CTA: tile t's maximum and its sum of exponentials relative to that
// maximum go to tile_m[t - t0] and tile_s[t - t0].  Returns whether this thread saw NaN or +inf.  The tiles are dealt
// out warp by warp, so that every warp has one before any has two; kNT of them are in flight per warp.
template <typename T>
__device__ __forceinline__ bool row_tile_stats(const T *zq, const Shape &s, int t0, int t1, float *tile_s, float *tile_m) {
    const int lane = threadIdx.x & 31, wid = warp_index(), nwarps = blockDim.x >> 5;
    bool bad = false;
    constexpr int kNT = 4;
    static_assert(kTile == 256, "a lane takes 8 entries of a tile");
    const bool pieces = (reinterpret_cast<uintptr_t>(zq) % 16 == 0) && (s.V % (16 / (int)sizeof(T)) == 0);
    for (int tb = t0 + wid; tb < t1; tb += nwarps * kNT) {
        float z[kNT][kTile / 32];
        if (pieces) {  // 16-byte loads
#pragma unroll
            for (int q = 0; q < kNT; ++q) load_tile_pieces<T>(zq, tb + q * nwarps, tb + q * nwarps < t1, s.V, lane, z[q]);
        } else {
#pragma unroll
            for (int q = 0; q < kNT; ++q)
#pragma unroll
                for (int e = 0; e < kTile / 32; ++e) {
                    const int x = (tb + q * nwarps) * kTile + lane + 32 * e;
                    z[q][e] = (tb + q * nwarps < t1 && x < s.V) ? ld_logit(zq, x) : -INFINITY;
                }
        }
        // the tiles are reduced side by side (independent shuffle chains), two entries per instruction
        float mt[kNT], acc[kNT];
#pragma unroll
        for (int q = 0; q < kNT; ++q) {
            mt[q] = -INFINITY;
#pragma unroll
            for (int e = 0; e < kTile / 32; e += 2) mt[q] = max3(mt[q], z[q][e], z[q][e + 1]);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
#pragma unroll
            for (int q = 0; q < kNT; ++q) mt[q] = fmaxf(mt[q], __shfl_xor_sync(0xffffffffu, mt[q], o));
#pragma unroll
        for (int q = 0; q < kNT; ++q) {
            // (a tile without a finite entry adds up zeros; what falls below 2^-126 of the tile's maximum adds nothing)
            const float2 nm = splat(mt[q] > -INFINITY ? -mt[q] : 0.0f), sc2 = splat(s.scale);
            float2 a2 = splat(0.0f);
#pragma unroll
            for (int e = 0; e < kTile / 32; e += 2) {
                const float2 v = __fmul2_rn(__fadd2_rn(make_float2(z[q][e], z[q][e + 1]), nm), sc2);
                a2 = __fadd2_rn(a2, make_float2(ex2(v.x), ex2(v.y)));
            }
            acc[q] = a2.x + a2.y;
            bad |= acc[q] != acc[q];  // NaN among the entries, or +inf (then inf - inf)
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
#pragma unroll
            for (int q = 0; q < kNT; ++q) acc[q] += __shfl_xor_sync(0xffffffffu, acc[q], o);
#pragma unroll
        for (int q = 0; q < kNT; ++q) {
            if (lane == 0 && tb + q * nwarps < t1) {
                tile_s[tb + q * nwarps - t0] = acc[q];
                tile_m[tb + q * nwarps - t0] = mt[q];
            }
        }
    }
    return bad;
}

__device__ __forceinline__ double warp_scan(double v, int lane) {
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const double up = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += up;
    }
    return v;
}

// Inverse CDF over tiles whose weights are known, by ONE warp and without a block barrier: every lane adds up a
// contiguous run of tiles, a scan over the lanes finds the run that the target (a mass) falls into, a second one the tile
// inside it, a third one the entry inside the tile (recomputed, 8 entries per lane).  weight(t): tile t's weight;
// entry(x): weight of entry x, which belongs to tile x / kTile - first_tile.  Where no entry's cumulative weight exceeds the
// target (rounding, or an infinite target), the last entry with positive weight of the part searched is taken.  All 32
// lanes must call and get the index (-1 if no tile has positive weight).
template <typename W, typename F>
__device__ __forceinline__ int warp_draw(W weight, int ntiles, int first_tile, int V, double target, F entry) {
    constexpr unsigned kAll = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const int per = (ntiles + 31) / 32;
    const int t0 = min(ntiles, lane * per), t1 = min(ntiles, t0 + per);
    double local = 0.0;
#pragma unroll 4
    for (int t = t0; t < t1; ++t) local += weight(t);
    double incl = warp_scan(local, lane);
    unsigned hit = uniform(__ballot_sync(kAll, local > 0.0 && incl > target));
    unsigned any = uniform(__ballot_sync(kAll, local > 0.0));
    if (any == 0u) return -1;
    int owner = hit ? __ffs(hit) - 1 : 31 - __clz(any);
    double base = __shfl_sync(kAll, incl - local, owner);
    const int r0 = owner * per, r1 = min(ntiles, r0 + per);
    int tile = -1, last = -1;
    for (int c0 = r0; c0 < r1 && tile < 0; c0 += 32) {
        const double v = c0 + lane < r1 ? weight(c0 + lane) : 0.0;
        incl = warp_scan(v, lane);
        hit = uniform(__ballot_sync(kAll, v > 0.0 && base + incl > target));
        any = uniform(__ballot_sync(kAll, v > 0.0));
        if (any) last = c0 + 31 - __clz(any);
        owner = hit ? __ffs(hit) - 1 : 31;
        if (hit) tile = c0 + owner;
        base += __shfl_sync(kAll, hit ? incl - v : incl, owner);
    }
    const bool crossed = tile >= 0;
    if (!crossed) tile = last;
    constexpr int kPer = kTile / 32;
    const int x0 = (first_tile + tile) * kTile + lane * kPer;
    float w[kPer];
    local = 0.0;
#pragma unroll
    for (int e = 0; e < kPer; ++e) {
        w[e] = x0 + e < V ? entry(x0 + e) : 0.0f;
        local += (double)w[e];
    }
    double cum = base + warp_scan(local, lane) - local;
    int first = -1;
    last = -1;
#pragma unroll
    for (int e = 0; e < kPer; ++e) {
        cum += (double)w[e];
        if (w[e] > 0.0f) {
            last = x0 + e;
            if (first < 0 && crossed && cum > target) first = x0 + e;
        }
    }
    hit = uniform(__ballot_sync(kAll, first >= 0));
    if (hit) return __shfl_sync(kAll, first, __ffs(hit) - 1);
    any = __ballot_sync(kAll, last >= 0);
    return any ? __shfl_sync(kAll, last, 31 - __clz(any)) : -1;
}

// What the CTAs of a cluster tell one another about their shares of a row (one double-word triple per CTA).
struct RowShare {
    double m, sum, bad;
};
constexpr int kMaxRowCtas = 8;
struct DrawScratch {
    RowShare share[kMaxRowCtas];
};
struct Drawn {
    int y;       // the entry, or -1: on the CTA that holds it only, and on rank 0 with `bad`
    bool bad;    // the row holds NaN or +inf, or no finite entry (every CTA)
    double total;  // the row's sum of exponentials relative to m
    float m;     // row maximum
};

// One token from softmax(zq/T) of a row by a cluster of C CTAs (C = 1: one CTA, no cluster needed), one pass over memory:
// every CTA takes `per` tiles (their statistics to tile_s, tile_m: `per` floats each), its first warp adds them up relative
// to the CTA's maximum and tells the other CTAs; the CTA whose share the target falls into searches its tiles and
// recomputes one.  All threads must call; warp 0's threads get the result, the other warps' y is undefined.  Every CTA of
// the cluster must be running (C > 1: the caller's cluster barrier).
template <typename T>
__device__ __forceinline__ Drawn draw_row(const T *zq, const Shape &s, double us, int rank, int C, float *tile_s, float *tile_m,
                                          DrawScratch *sc) {
    const int lane = threadIdx.x & 31, wid = warp_index();
    const int per = (s.ntiles + C - 1) / C, t0 = min(s.ntiles, rank * per), t1 = min(s.ntiles, t0 + per);
    const bool mybad = row_tile_stats<T>(zq, s, t0, t1, tile_s, tile_m);
    const bool anybad = __syncthreads_or(mybad);
    Drawn o{-1, true, 0.0, -INFINITY};
    float m = -INFINITY;
    double S = 0.0;
    if (wid == 0) {
        for (int t = lane; t < t1 - t0; t += 32) m = fmaxf(m, tile_m[t]);
        m = warp_max(m);
        if (m > -INFINITY)
            for (int t = lane; t < t1 - t0; t += 32)
                S += tile_m[t] > -INFINITY ? (double)tile_s[t] * (double)expo(tile_m[t], m, s.scale) : 0.0;
        S = warp_sum(S);
        if (C > 1 && lane < C) {
            st_peer(&sc->share[rank].m, lane, (double)m);
            st_peer(&sc->share[rank].sum, lane, S);
            st_peer(&sc->share[rank].bad, lane, anybad ? 1.0 : 0.0);
        }
    }
    if (C > 1) {
        cluster_arrive();
        cluster_wait();
    }
    if (wid > 0) return o;
    // the CTAs' shares, rank by rank (= in vocabulary order), in units of the row maximum
    double mass = S, factor = 1.0, before = 0.0;
    bool bad = anybad;
    o.m = m;
    if (C > 1) {
        const RowShare sh = lane < C ? sc->share[lane] : RowShare{-INFINITY, 0.0, 0.0};
        o.m = warp_max((float)sh.m);
        bad = __any_sync(0xffffffffu, sh.bad != 0.0);
        const double f = (float)sh.m > -INFINITY ? exp2_short((sh.m - (double)o.m) * (double)s.scale) : 0.0;
        mass = sh.sum * f;
        factor = __shfl_sync(0xffffffffu, f, rank);
        double run = 0.0;
        int owner = -1, last = -1;
        for (int r = 0; r < C; ++r) o.total += __shfl_sync(0xffffffffu, mass, r);
        const double target = us * o.total;
        for (int r = 0; r < C; ++r) {
            const double v = __shfl_sync(0xffffffffu, mass, r);
            if (v > 0.0) last = r;
            if (owner < 0 && run + v > target) owner = r;
            if (r < rank) before += v;
            run += v;
        }
        o.bad = bad || !(o.m > -INFINITY);
        owner = uniform(owner);
        last = uniform(last);
        o.bad = uniform((int)o.bad) != 0;
        if (o.bad || rank != (owner < 0 ? last : owner)) return o;
        if (owner < 0) before = -INFINITY;  // no share crosses: its last entry with positive weight
    } else {
        o.total = S;
        o.bad = uniform((int)(bad || !(o.m > -INFINITY))) != 0;
        if (o.bad) return o;
    }
    auto weight = [&](int t) { return tile_m[t] > -INFINITY ? (double)tile_s[t] * (double)expo(tile_m[t], m, s.scale) : 0.0; };
    auto entry = [&](int x) { return expo(ld_logit(zq, x), m, s.scale); };
    o.y = warp_draw(weight, t1 - t0, t0, s.V, (us * o.total - before) / factor, entry);
    return o;
}

// One token from softmax(zq/T) of a single row in one pass over memory: every tile's maximum and its sum of
// exponentials relative to that maximum, then the row maximum, the factors that move the tile sums to it, the
// tile search and the pick inside the tile.  tile_s, tile_m: ntiles floats each (shared or global scratch).
// Returns the token, or -1 with `bad` set if the row holds NaN/+inf or no finite logit.  On return tile_s[t] * tile_m[t]
// is tile t's sum of exponentials relative to the row maximum.  All threads must call.
template <typename T>
__device__ int draw_from_row(const T *zq, const Shape &s, double us, float *tile_s, float *tile_m, SampleScratch *sc,
                             bool &bad_out) {
    const int tid = threadIdx.x, lane = tid & 31;
    const int nthreads = blockDim.x;
    const bool bad = __syncthreads_or(row_tile_stats<T>(zq, s, 0, s.ntiles, tile_s, tile_m));
    float m = -INFINITY;  // (every warp for itself)
    for (int t = lane; t < s.ntiles; t += 32) m = fmaxf(m, tile_m[t]);
    m = warp_max(m);
    if (bad || !(m > -INFINITY)) {
        bad_out = true;
        return -1;
    }
    bad_out = false;
    __syncthreads();  // every warp has read the maxima
    // tile_m becomes the factor exp((m_t - m)/T) of its tile
    for (int t = tid; t < s.ntiles; t += nthreads) tile_m[t] = (tile_m[t] > -INFINITY) ? expo(tile_m[t], m, s.scale) : 0.0f;
    __syncthreads();
    // the target is us times the row's total, which the tile search computes on its way
    locate_tile(tile_s, tile_m, s.ntiles, us, true, sc->i, sc->d, sc->warp);
    const int sel = sc->i[2];
    const int x0 = sel * kTile, x1 = min(s.V, x0 + kTile);
    auto wfun = [&](int x) { return expo(ld_logit(zq, x), m, s.scale); };
    Pick p = pick_in_tile(x0, x1, sc->d[0], sc->d[1], wfun, sc->warp, sc->pick);
    return (p.first != INT_MAX) ? p.first : p.last;
}

}  // namespace sgbv
