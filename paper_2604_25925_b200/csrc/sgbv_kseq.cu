// Comparison verifiers of Section 3 of the paper, behind the same boundary as the block verifier:
// SpecTr's position-wise K-SEQ (Section 3.2) and, as its one-draft case, token-level speculative sampling
// (Section 3.1).  They exist so that the verification cost of the methods can be compared on one machine
// (the paper's Table 2).
//
// One cluster of C CTAs per batch row walks the positions i = 0..gamma-1 in order.  At a position the drafts that still
// match the accepted prefix ("retained", n of them) are the candidates; they share the rows of that prefix, and the
// rows of the first retained draft are read:
//   1. every CTA reads its share of the target and the draft row ONCE into shared memory; row maxima, then the
//      exponentials in place and their sums, both exchanged within the cluster;
//   2. rho in [1, n]: root of 1 - (1 - beta(rho))^n = rho beta(rho), beta(rho) = sum_x min{p(x), q(x)/rho}.  With the excess
//      E(rho) = sum_x max{q(x) - rho p(x), 0} it reads E = (1 - beta)^n, 1 - beta = (E + rho - 1) / rho: nothing cancels however
//      close the rows are.  Newton's method from the exponentials in shared memory, inside a bracket that every step shrinks;
//      one sweep gives E and the slope (n = 1: rho = 1);
//   3. the retained drafts are tried in order, draft k's token x is accepted if eta < min{1, q(x)/(rho p(x))};
//      the first accepted token extends the prefix, the drafts with that token stay retained;
//   4. if none is accepted: y from norm(max{q - rho p, 0}) by inverse CDF over per-tile sums, and the row is done.
// After gamma accepted positions y is drawn from the target row that follows the block.  All decisions are taken by every
// CTA of the cluster from the same numbers.
//
// What bounds it is the serial chain: positions one after the other, some seven sweeps and as many cluster exchanges each
// (five for rho on ordinary rows, up to some 30 where target and draft nearly agree).  Rows stay on chip between the sweeps (a
// CTA holds up to kCapTiles tiles; the rest of a longer share is read again in every sweep), and a row is spread over as many
// CTAs as the batch leaves free.  64 prompts, K = 3, gamma = 12, 32256 float32: 66-72 us from machine to machine (two prompts in
// three stop at the first or second position; the time is that of the longest walk), against 370-480 of one CTA of 1024 threads per
// prompt that read the rows from L2 in two sweeps for the statistics and one for each of 34 bisections.  With one draft
// there is no rho, and batches that leave no SM idle hold nothing (kHeld = false; the rule and its figures stand at run()).
#include <atomic>

#include "sgbv_sample.cuh"

namespace sgbv {

namespace {

constexpr int kThreads = 512;        // two CTAs per SM
constexpr int kWarpsPerCta = kThreads / 32;
constexpr int kSlots = 2 * 148;      // CTAs the device holds, of up to half of kCapTiles tiles (or none held); longer ones: half as many
constexpr int kCapTiles = 104;       // tiles of both rows in one CTA's shared memory (208 KB)
constexpr int kNewtonSteps = 40;     // sweeps that may follow Newton's method; then
constexpr int kMaxSteps = 80;        // as many that halve the bracket: n 2^-40 is left of it in any case

struct KseqScratch {
    double part[2][kWarpsPerCta];
    double slots[2][kMaxRowCtas][2];   // by parity of the exchange: every CTA's pair of values
    DrawScratch draw;
    float tiles[2][kCapTiles];
    int kept[kMaxK];
    int n, accepted;
};

// Two values per thread combined over the cluster (sum, or maximum); every thread of every CTA gets the results, and
// slots[par][r] keeps CTA r's share until the exchange after the next one.  All threads must call.
template <bool kMaximum, bool kHeld>
__device__ __forceinline__ void exchange(double &a, double &b, KseqScratch &sc, int rank, int C, int &par) {
    const int lane = threadIdx.x & 31, wid = warp_index();
    auto op = [](double x, double y) { return kMaximum ? fmax(x, y) : x + y; };
    auto all = [&](double v) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v = op(v, __shfl_xor_sync(0xffffffffu, v, o));
        return v;
    };
    a = all(a);
    b = all(b);
    if (lane == 0) {
        sc.part[0][wid] = a;
        sc.part[1][wid] = b;
    }
    __syncthreads();
    par ^= 1;
    if (wid == 0) {
        const double none = kMaximum ? -INFINITY : 0.0;
        a = all(lane < kWarpsPerCta ? sc.part[0][lane] : none);
        b = all(lane < kWarpsPerCta ? sc.part[1][lane] : none);
        if (lane < C) {
            st_peer(&sc.slots[par][rank][0], lane, a);
            st_peer(&sc.slots[par][rank][1], lane, b);
        }
    }
    if (kHeld || C > 1) {
        cluster_arrive();
        cluster_wait();
    } else {
        __syncthreads();
    }
    a = sc.slots[par][0][0];
    b = sc.slots[par][0][1];
    for (int r = 1; r < C; ++r) {  // (rank order: the same on every CTA)
        a = op(a, sc.slots[par][r][0]);
        b = op(b, sc.slots[par][r][1]);
    }
}

// f(8 target logits, 8 draft logits) over the entries of tiles t0..t1-1 of a pair of rows, by the whole CTA (-inf in the places
// past the end): in 16-byte pieces, two tiles of both rows in flight per warp, where the rows can be read so.
template <typename T, typename F>
__device__ __forceinline__ void for_entries(const T *zq, const T *zp, int t0, int t1, int V, bool pieces, F f) {
    constexpr int kPer = kTile / 32;
    if (!pieces) {
        const int end = min(V, t1 * kTile);
        int x = t0 * kTile + threadIdx.x;
        float a[kPer], c[kPer];
        for (; x + (kPer - 1) * kThreads < end; x += kPer * kThreads) {
#pragma unroll
            for (int e = 0; e < kPer; ++e) {
                a[e] = ld_logit(zq, x + e * kThreads);
                c[e] = ld_logit(zp, x + e * kThreads);
            }
            f(a, c);
        }
#pragma unroll
        for (int e = 0; e < kPer; ++e) {
            const bool in = x + e * kThreads < end;
            a[e] = in ? ld_logit(zq, x + e * kThreads) : -INFINITY;
            c[e] = in ? ld_logit(zp, x + e * kThreads) : -INFINITY;
        }
        f(a, c);
        return;
    }
    const int lane = threadIdx.x & 31;
    for (int t = t0 + warp_index(); t < t1; t += 2 * kWarpsPerCta) {
        float a[2][kPer], c[2][kPer];
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const int tt = t + q * kWarpsPerCta;
            load_tile_pieces<T>(zq, tt, tt < t1, V, lane, a[q]);
            load_tile_pieces<T>(zp, tt, tt < t1, V, lane, c[q]);
        }
#pragma unroll
        for (int q = 0; q < 2; ++q) f(a[q], c[q]);
    }
}

// kHeld: the CTA keeps the exponentials of its tiles in shared memory.  Without it (one draft: nothing but the normalisers is
// added up, so a row is gone through twice and, once per prompt, a third time) it has none, and two CTAs share an SM at any length.
template <typename T, bool kHeld>
__global__ void __launch_bounds__(kThreads, 2)
kseq_kernel(const T *__restrict__ zq_all, const T *__restrict__ zp_all, const int32_t *__restrict__ tok_all,
            const float *__restrict__ u_all, Shape s, int C, float *__restrict__ tile_scratch, int32_t *__restrict__ out_tau,
            int32_t *out_tokens, double *__restrict__ out_rho, double *__restrict__ out_acc,
            int32_t *__restrict__ out_status) {
    extern __shared__ __align__(16) float rows_s[];  // exponentials of this CTA's tiles: target row, then draft row
    __shared__ KseqScratch sc;
    const int rank = (int)cluster_ctarank();
    cluster_arrive();
    const int b = blockIdx.x / C, tid = threadIdx.x, lane = tid & 31, wid = warp_index();
    const int K = s.K, g = s.gamma, V = s.V;
    const int32_t *tok = tok_all + (size_t)b * K * g;
    const float *u = u_all + (size_t)b * (K * g + 1);
    const int per = (s.ntiles + C - 1) / C, t0 = min(s.ntiles, rank * per), t1 = min(s.ntiles, t0 + per);
    const int held = kHeld ? min(t1 - t0, kCapTiles) : 0;  // tiles in shared memory
    const int rest0 = (t0 + held) * kTile, rest1 = min(V, t1 * kTile);  // entries that are read again in every sweep
    float *eq_s = rows_s, *ep_s = rows_s + (size_t)min(per, kCapTiles) * kTile;
    // per-tile sums: in shared memory, or for long shares in global scratch
    float *tile_s = sc.tiles[0], *tile_m = sc.tiles[1];
    if (per > kCapTiles) {
        tile_s = tile_scratch + (size_t)b * 2 * s.ntiles + t0;
        tile_m = tile_s + s.ntiles;
    }
    const bool lead = rank == 0 && tid == 0;

    if (rank == 0) {
        for (int n = tid; n <= g; n += kThreads) out_tokens[(size_t)b * (g + 1) + n] = -1;
        if (out_rho)
            for (int n = tid; n < g; n += kThreads) out_rho[(size_t)b * g + n] = NAN;
        if (out_acc)
            for (int n = tid; n < K * g; n += kThreads) out_acc[(size_t)b * K * g + n] = NAN;
    }
    if (tid == 0) sc.n = K;
    for (int k = tid; k < K; k += kThreads) sc.kept[k] = k;
    bool range = false;
    for (int n = tid; n < K * g; n += kThreads) range |= tok[n] < 0 || tok[n] >= V;
    range = __syncthreads_or(range);
    cluster_wait();  // every CTA of the cluster is running
    if (range) {
        if (lead) {
            out_tau[b] = -1;
            out_status[b] = SGBV_STATUS_TOKEN_RANGE;
        }
        return;
    }

    int tau = 0, flags = 0, par = 0;
    bool stopped = false;
    for (int i = 0; i < g && !stopped; ++i) {
        const int k0 = uniform(sc.kept[0]), nk = uniform(sc.n);
        const T *zq = zq_all + (((size_t)b * K + k0) * (g + 1) + i) * V;
        const T *zp = zp_all + (((size_t)b * K + k0) * g + i) * V;
        // the logits of the retained drafts' tokens, fetched ahead (first warp, two drafts per lane)
        float zqx[2] = {0.0f, 0.0f}, zpx[2] = {0.0f, 0.0f};
        int tokx[2] = {-1, -1};
        if (wid == 0)
#pragma unroll
            for (int e = 0; e < 2; ++e)
                if (lane + 32 * e < nk) {
                    tokx[e] = tok[sc.kept[lane + 32 * e] * g + i];
                    zqx[e] = ld_logit(zq, tokx[e]);
                    zpx[e] = ld_logit(zp, tokx[e]);
                }
        // ---- 1. logits to shared memory, maxima; exponentials, normalisers ---------------------------------
        const bool pieces = (reinterpret_cast<uintptr_t>(zq) % 16 == 0) && (reinterpret_cast<uintptr_t>(zp) % 16 == 0) &&
                            (V % (16 / (int)sizeof(T)) == 0);
        float mqf = -INFINITY, mpf = -INFINITY;
        for (int t = wid; t < held; t += 2 * kWarpsPerCta) {  // two tiles of both rows in flight per warp
            float a[2][kTile / 32], c[2][kTile / 32];
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                const int tt = t + q * kWarpsPerCta;
                if (pieces) {
                    load_tile_pieces<T>(zq, t0 + tt, tt < held, V, lane, a[q]);
                    load_tile_pieces<T>(zp, t0 + tt, tt < held, V, lane, c[q]);
                } else {
#pragma unroll
                    for (int e = 0; e < kTile / 32; ++e) {
                        const int x = (t0 + tt) * kTile + lane + 32 * e;
                        a[q][e] = tt < held && x < V ? ld_logit(zq, x) : -INFINITY;
                        c[q][e] = tt < held && x < V ? ld_logit(zp, x) : -INFINITY;
                    }
                }
            }
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                const int tt = t + q * kWarpsPerCta;
                if (tt >= held) break;
#pragma unroll
                for (int e = 0; e < kTile / 32; ++e) {
                    mqf = fmaxf(mqf, a[q][e]);
                    mpf = fmaxf(mpf, c[q][e]);
                }
                float *dq = eq_s + tt * kTile, *dp = ep_s + tt * kTile;
                if (pieces) {
                    // where load_tile_pieces takes a lane's entries from
                    const int xa = sizeof(T) == 4 ? lane * 4 : lane * 8, xb = sizeof(T) == 4 ? kTile / 2 + lane * 4 : lane * 8 + 4;
                    *reinterpret_cast<float4 *>(dq + xa) = make_float4(a[q][0], a[q][1], a[q][2], a[q][3]);
                    *reinterpret_cast<float4 *>(dq + xb) = make_float4(a[q][4], a[q][5], a[q][6], a[q][7]);
                    *reinterpret_cast<float4 *>(dp + xa) = make_float4(c[q][0], c[q][1], c[q][2], c[q][3]);
                    *reinterpret_cast<float4 *>(dp + xb) = make_float4(c[q][4], c[q][5], c[q][6], c[q][7]);
                } else {
#pragma unroll
                    for (int e = 0; e < kTile / 32; ++e) {
                        dq[lane + 32 * e] = a[q][e];
                        dp[lane + 32 * e] = c[q][e];
                    }
                }
            }
        }
        if (kHeld) {
            for (int x = rest0 + tid; x < rest1; x += kThreads) {
                mqf = fmaxf(mqf, ld_logit(zq, x));
                mpf = fmaxf(mpf, ld_logit(zp, x));
            }
        } else {
            for_entries<T>(zq, zp, t0, t1, V, pieces, [&](const float (&a)[8], const float (&c)[8]) {
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    mqf = fmaxf(mqf, a[e]);
                    mpf = fmaxf(mpf, c[e]);
                }
            });
        }
        double mqd = (double)mqf, mpd = (double)mpf;
        exchange<true, kHeld>(mqd, mpd, sc, rank, C, par);
        const float mq = (float)mqd, mp = (float)mpd;
        const float nmq = mq > -INFINITY ? -mq : 0.0f, nmp = mp > -INFINITY ? -mp : 0.0f;
        auto eqof = [&](float z) { return ex2((z + nmq) * s.scale); };
        auto epof = [&](float z) { return ex2((z + nmp) * s.scale); };
        float4 *const eq4 = reinterpret_cast<float4 *>(eq_s), *const ep4 = reinterpret_cast<float4 *>(ep_s);
        const int n4 = held * (kTile / 4);
        float sq = 0.0f, sp = 0.0f;
        for (int j = tid; j < n4; j += kThreads) {
            float4 a = eq4[j], c = ep4[j];
            a = make_float4(eqof(a.x), eqof(a.y), eqof(a.z), eqof(a.w));
            c = make_float4(epof(c.x), epof(c.y), epof(c.z), epof(c.w));
            eq4[j] = a;
            ep4[j] = c;
            sq += (a.x + a.y) + (a.z + a.w);
            sp += (c.x + c.y) + (c.z + c.w);
        }
        if (kHeld) {
            for (int x = rest0 + tid; x < rest1; x += kThreads) {
                sq += eqof(ld_logit(zq, x));
                sp += epof(ld_logit(zp, x));
            }
        } else {
            // (eight at a time, in a tree: short chains of float32 additions)
            auto sum8 = [](float a, float b, float c, float d, float e, float f, float g, float h) {
                return ((a + b) + (c + d)) + ((e + f) + (g + h));
            };
            for_entries<T>(zq, zp, t0, t1, V, pieces, [&](const float (&a)[8], const float (&c)[8]) {
                sq += sum8(eqof(a[0]), eqof(a[1]), eqof(a[2]), eqof(a[3]), eqof(a[4]), eqof(a[5]), eqof(a[6]), eqof(a[7]));
                sp += sum8(epof(c[0]), epof(c[1]), epof(c[2]), epof(c[3]), epof(c[4]), epof(c[5]), epof(c[6]), epof(c[7]));
            });
        }
        double Zq = (double)sq, Zp = (double)sp;
        exchange<false, kHeld>(Zq, Zp, sc, rank, C, par);
        // NaN entries end up in the sums; +inf is its row's maximum and gives inf - inf there
        if (uniform((int)(!(mq > -INFINITY) || !(mp > -INFINITY) || Zq != Zq || Zp != Zp))) {
            flags |= SGBV_STATUS_NONFINITE_LOGIT;
            break;
        }
        // ---- 2. rho (the same on every thread of the cluster) ----------------------------------------------
        double rho = 1.0;
        if (kHeld && nk > 1) {
            double lo = 1.0, hi = (double)nk;
            for (int it = 0; it < kMaxSteps; ++it) {
                const double r = rho * (Zq / Zp);
                const float thr = (float)r;
                float e = 0.0f, s2 = 0.0f;  // sums over the entries with q > rho p: of q - thr p and of p
                auto excess = [&](float a, float c) { return fmaxf(fmaf(-thr, c, a), 0.0f); };
                auto p_of = [&](float d, float c) { return d > 0.0f ? c : 0.0f; };
                for (int j = tid; j < n4; j += kThreads) {
                    const float4 a = eq4[j], c = ep4[j];
                    const float dx = excess(a.x, c.x), dy = excess(a.y, c.y), dz = excess(a.z, c.z), dw = excess(a.w, c.w);
                    e += (dx + dy) + (dz + dw);
                    s2 += (p_of(dx, c.x) + p_of(dy, c.y)) + (p_of(dz, c.z) + p_of(dw, c.w));
                }
                for (int x = rest0 + tid; x < rest1; x += kThreads) {
                    const float c = epof(ld_logit(zp, x)), d = excess(eqof(ld_logit(zq, x)), c);
                    e += d;
                    s2 += p_of(d, c);
                }
                double E = (double)e, S2 = (double)s2;
                exchange<false, kHeld>(E, S2, sc, rank, C, par);
                E = fmax(E - (r - (double)thr) * S2, 0.0) / Zq;  // (thr is the float32 next to r)
                S2 /= Zp;
                const double miss = fmax(E + (rho - 1.0), 0.0) / rho;  // 1 - beta
                double pw = 1.0;
                for (int j = 1; j < nk; ++j) pw *= miss;
                const double f = E - pw * miss;
                if (f > 0.0) lo = rho;
                else hi = rho;
                if (uniform((int)(hi <= lo))) break;  // (f <= 0 at 1: the root is 1)
                const double S1 = fmax(1.0 - E - rho * S2, 0.0);
                const double df = -(double)nk * pw * S1 / (rho * rho) - S2;
                double next = rho - f / df;
                // (right of the largest q / p nothing is left of E, and Newton's method would creep back)
                const bool creeps = it >= kNewtonSteps || !(S2 > 0.0);
                // the last step: below the resolution of the float32 sums (asked before the bracket is: the step may be 0)
                const bool last = !creeps && fabs(next - rho) <= 1e-8 * rho;
                if (!last && (creeps || !(next > lo && next < hi))) next = 0.5 * (lo + hi);
                rho = fmin(fmax(next, lo), hi);
                if (uniform((int)(last || hi - lo <= 1e-8 * rho))) break;
            }
        }
        // ---- 3. the retained drafts, in order (first warp of every CTA) -----------------------------------------
        if (wid == 0) {
            if (lead && out_rho) out_rho[(size_t)b * g + i] = rho;
            const double lZq = log(Zq), lZp = log(Zp);
            double acc[2];
            unsigned pass[2];
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const int j = lane + 32 * e;
                acc[e] = 1.0;
                if (j < nk && zpx[e] > -INFINITY) {
                    const double lq = ((double)zqx[e] - (double)mq) * s.inv_T - lZq;
                    const double lp = ((double)zpx[e] - (double)mp) * s.inv_T - lZp;
                    acc[e] = exp(lq - lp) / rho;
                    if (!(acc[e] < 1.0)) acc[e] = 1.0;
                }
                pass[e] = __ballot_sync(0xffffffffu, j < nk && (double)u[(j < nk ? sc.kept[j] : 0) * g + i] < acc[e]);
            }
            const int first = pass[0] ? __ffs(pass[0]) - 1 : pass[1] ? 31 + __ffs(pass[1]) : -1;  // among the retained
            const int x = first < 0 ? -1 : __shfl_sync(0xffffffffu, first < 32 ? tokx[0] : tokx[1], first & 31);
            int stay[2], m = 0;
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const int j = lane + 32 * e, k = j < nk ? sc.kept[j] : 0;
                if (rank == 0 && out_acc && j < nk && (first < 0 || j <= first)) out_acc[((size_t)b * K + k) * g + i] = acc[e];
                const unsigned same = __ballot_sync(0xffffffffu, first >= 0 && j < nk && tokx[e] == x);
                stay[e] = (same >> lane) & 1u ? m + __popc(same & ((1u << lane) - 1u)) : -1;
                tokx[e] = k;  // (the draft)
                m += __popc(same);
            }
            __syncwarp();
#pragma unroll
            for (int e = 0; e < 2; ++e)
                if (stay[e] >= 0) sc.kept[stay[e]] = tokx[e];
            if (lane == 0) {
                sc.accepted = first;
                if (first >= 0) {
                    sc.n = m;
                    if (rank == 0) out_tokens[(size_t)b * (g + 1) + i] = x;
                }
            }
        }
        __syncthreads();
        if (uniform(sc.accepted) >= 0) {
            tau = i + 1;
            continue;
        }
        // ---- 4. nothing accepted: y from norm(max{q - rho p, 0}) ------------------------------------------------
        stopped = true;
        const float iZq = (float)(1.0 / Zq), rho_p = (float)rho * (float)(1.0 / Zp);
        auto wof = [&](float a, float c) { return fmaxf(a * iZq - c * rho_p, 0.0f); };
        // (exp2f: ex2 flushes what lies below 2^-126 of the row's maximum to 0)
        auto eq_full = [&](int x) { return exp2f((ld_logit(zq, x) + nmq) * s.scale); };
        auto ep_full = [&](int x) { return exp2f((ld_logit(zp, x) + nmp) * s.scale); };
        auto entry = [&](int x) {
            const int j = x - t0 * kTile;
            return j < held * kTile ? wof(eq_s[j], ep_s[j]) : wof(eq_full(x), ep_full(x));
        };
        double W = 0.0;
        for (bool full = !kHeld;; full = true) {
            for (int t = wid; t < t1 - t0; t += kWarpsPerCta) {  // one warp per tile
                float acc = 0.0f;
#pragma unroll
                for (int e = 0; e < kTile / 32; ++e) {
                    const int x = (t0 + t) * kTile + lane + 32 * e;
                    if (x < V) acc += entry(x);
                }
                acc = warp_sum(acc);
                if (lane == 0) tile_s[t] = acc;
            }
            __syncthreads();
            double unused = 0.0;
            W = 0.0;
            for (int t = tid; t < t1 - t0; t += kThreads) W += (double)tile_s[t];
            exchange<false, kHeld>(W, unused, sc, rank, C, par);
            if (full || uniform((int)(W > 0x1p-90))) break;
            // next to no mass: what was flushed may be all there is of q - rho p, so the held exponentials are made again
            for (int j = tid; j < held * kTile; j += kThreads)
                if (t0 * kTile + j < V) {
                    eq_s[j] = eq_full(t0 * kTile + j);
                    ep_s[j] = ep_full(t0 * kTile + j);
                }
            __syncthreads();
        }
        const double us = (double)u[K * g];
        if (uniform((int)(W > 0.0))) {
            // the CTA whose share the target falls into draws
            const double target = us * W;
            double run = 0.0, before = 0.0;
            int owner = -1, last = -1;
            for (int r = 0; r < C; ++r) {
                const double v = sc.slots[par][r][0];
                if (v > 0.0) last = r;
                if (owner < 0 && run + v > target) owner = r;
                if (r < rank) before += v;
                run += v;
            }
            if (rank == uniform(owner < 0 ? last : owner) && wid == 0) {
                auto weight = [&](int t) { return (double)tile_s[t]; };
                const int y = warp_draw(weight, t1 - t0, t0, V, owner < 0 ? INFINITY : target - before, entry);
                if (lane == 0) out_tokens[(size_t)b * (g + 1) + i] = y;
            }
        } else {  // q <= rho p everywhere: the draw comes from q itself
            flags |= SGBV_STATUS_DEGENERATE_RESIDUAL;
            const Drawn d = draw_row<T>(zq, s, us, rank, C, tile_s, tile_m, &sc.draw);
            if (tid == 0 && d.y >= 0) out_tokens[(size_t)b * (g + 1) + i] = d.y;
        }
    }
    if (!stopped && !(flags & SGBV_STATUS_NONFINITE_LOGIT)) {  // every position accepted: bonus token
        const T *zq = zq_all + (((size_t)b * K + sc.kept[0]) * (g + 1) + g) * V;
        const Drawn d = draw_row<T>(zq, s, (double)u[K * g], rank, C, tile_s, tile_m, &sc.draw);
        if (wid == 0 && d.bad) flags |= SGBV_STATUS_NONFINITE_LOGIT;  // (the first warps know)
        if (tid == 0 && d.y >= 0) out_tokens[(size_t)b * (g + 1) + g] = d.y;
    }
    if (rank == 0 && wid == 0) {
        const bool failed = (flags & SGBV_STATUS_NONFINITE_LOGIT) != 0;
        if (failed)
            for (int n = lane; n <= g; n += 32) out_tokens[(size_t)b * (g + 1) + n] = -1;
        if (lane == 0) {
            out_tau[b] = failed ? -1 : tau;
            out_status[b] = flags;
        }
    }
}

template <typename T, bool kHeld>
int run_as(const Launch &L, int C, float *tile_scratch, double *out_rho, double *out_acc, int32_t *out_status) {
    const Shape &s = L.s;
    int dev = 0;
    static std::atomic<bool> attr_done[64];
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return SGBV_ERR_CUDA;
    if (kHeld && !attr_done[dev]) {
        if (cudaFuncSetAttribute(kseq_kernel<T, kHeld>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 2 * kCapTiles * kTile * (int)sizeof(float)) != cudaSuccess)
            return SGBV_ERR_CUDA;
        attr_done[dev] = true;
    }
    const int per = (s.ntiles + C - 1) / C;
    const size_t smem = kHeld ? 2 * (size_t)(per < kCapTiles ? per : kCapTiles) * kTile * sizeof(float) : 0;
    if (launch_clusters(kseq_kernel<T, kHeld>, (unsigned)s.B * (unsigned)C, kThreads, smem, C, L.stream, (const T *)L.zq,
                        (const T *)L.zp, L.tok, L.u, s, C, tile_scratch, L.out_tau, L.out_tokens, out_rho, out_acc,
                        out_status) == cudaSuccess)
        return 1;
    cudaGetLastError();
    return SGBV_ERR_CUDA;
}

template <typename T>
int run(const Launch &L, float *tile_scratch, double *out_rho, double *out_acc, int32_t *out_status) {
    const Shape &s = L.s;
    // as few CTAs as hold a row on chip; more while the device has room for all of the batch's and a CTA keeps a tile for
    // every other warp
    int C = 1;
    while (C < kMaxRowCtas && (s.ntiles > C * kCapTiles ||
                               ((long)s.B * 2 * C <= kSlots && s.ntiles >= 2 * C * (kWarpsPerCta / 2))))
        C *= 2;
    // One draft has no sums to add up again and again: holding its rows only pays while the CTAs are all resident (one per SM where
    // a share is longer than half of kCapTiles), and a row of a few tiles is done before a cluster has met.  Else nothing is
    // held: one CTA for 128 KB of a row, two for 256, four beyond, more while the device has room for the batch's and a CTA
    // keeps 28 tiles.  us, gamma = 4, held : not held (one CTA of 1024 threads per prompt and no cluster): 1024 prompts of 128256
    // bfloat16 1563 : 656 (915), 148 of them 258 : 127 (215); 148 of 50257 110 : 71 (81), float32 108 : 82 (96); 400 of 32256 float32
    // 149 : 131 (146); 148 of 8192 33 : 27 (31).
    const int per = (s.ntiles + C - 1) / C;
    const bool resident = per <= kCapTiles / 2 || (long)s.B * C <= (C == kMaxRowCtas ? 3 * kSlots / 4 : kSlots / 2);
    if (s.K == 1 && (s.ntiles <= 32 || s.B > kSlots / 2 || !resident)) {
        const size_t bytes = (size_t)s.V * sizeof(T);
        C = bytes <= 128 * 1024 ? 1 : bytes <= 256 * 1024 ? 2 : 4;
        while (C < kMaxRowCtas && (long)s.B * 2 * C <= kSlots && s.ntiles >= 2 * C * 28) C *= 2;
        return run_as<T, false>(L, C, tile_scratch, out_rho, out_acc, out_status);
    }
    return run_as<T, true>(L, C, tile_scratch, out_rho, out_acc, out_status);
}

}  // namespace

int launch_kseq(const Launch &L, float *tile_scratch, double *out_rho, double *out_acc, int32_t *out_status) {
    return L.dtype == SGBV_DTYPE_BF16 ? run<uint16_t>(L, tile_scratch, out_rho, out_acc, out_status)
                                      : run<float>(L, tile_scratch, out_rho, out_acc, out_status);
}

}  // namespace sgbv
