// dm_choice.cu -- the SLO-aware choice (Sec. 3.2; App. A.1.1: TTFT(r,i) =
// T_q(r,i) + T_c(r,i)), the rules it is compared with (Sec. 2.2, Sec. 4.3),
// and the serving metrics sampled at choice time (Sec. 2.2 CV; Sec. 4.1).
//
// Queues: instance i owns a ring buffer of Q entries with monotonically
// increasing head/tail counters; W[i] is the sum of remaining work.
//
// Choice between two candidates (DualMap's rule and the pair variants):
// the decision for a request depends on the loads left by every earlier
// request of the batch that shares one of its candidates.  One CTA keeps W
// in shared memory; one warp decides 32 requests at a time, level by level (a
// request follows only the earlier requests of the window that share an
// instance with it); everything that does not depend on W is precomputed
// in parallel, and queue writes and outputs are emitted in parallel
// afterwards.
//
// Cluster-wide rules: every request depends on every earlier one, so one
// warp decides them one at a time (an argmin over the live instances),
// with the hits on every live instance probed beforehand by k_probe_all.
//
// At the end of the file: routing with d candidates (App. A.8).
#include <algorithm>
#include <atomic>
#include <type_traits>

#include "dm_internal.cuh"
#include "dm_run_end.h"

namespace dm {

// ---------------------------------------------------------------------------
// Block-wide helpers of the single-CTA choice kernels (1024 threads).

__device__ __forceinline__ unsigned __int128 shfl_xor_u128(unsigned __int128 v, int o) {
    const uint64_t lo = shfl_xor_u64((uint64_t)v, o), hi = shfl_xor_u64((uint64_t)(v >> 64), o);
    return ((unsigned __int128)hi << 64) | lo;
}

struct MetricSums {
    uint64_t tokens, hits, sw, est;
};

// Sums each thread's per-request counters and this thread's share of the
// live instances' S1 = sum W, S2 = sum W^2 and count over the block; one
// thread adds the counters to the metrics (fire-and-forget atomics) and
// leaves the sums as the batch's pending CV sample.  Called by all threads.
__device__ void finish_metrics(const DevState &d, uint32_t n, MetricSums ms, unsigned __int128 S1,
                               unsigned __int128 S2, uint32_t cnt) {
    __shared__ unsigned long long s_u[32][5];
    __shared__ unsigned __int128 s_w[32][2];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    uint64_t v[5] = {ms.tokens, ms.hits, ms.sw, ms.est, cnt};
#pragma unroll
    for (int j = 0; j < 5; ++j) v[j] = warp_sum_u64(v[j]);
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) {
        S1 += shfl_xor_u128(S1, o);
        S2 += shfl_xor_u128(S2, o);
    }
    if (lane == 0) {
#pragma unroll
        for (int j = 0; j < 5; ++j) s_u[wid][j] = v[j];
        s_w[wid][0] = S1;
        s_w[wid][1] = S2;
    }
    __syncthreads();
    if (wid == 0) {
        // lane w takes warp w's partials; one more warp reduction
        const int nw = (blockDim.x + 31) >> 5;
        uint64_t t[5];
#pragma unroll
        for (int j = 0; j < 5; ++j) t[j] = warp_sum_u64(lane < nw ? s_u[lane][j] : 0);
        unsigned __int128 a = lane < nw ? s_w[lane][0] : 0, b = lane < nw ? s_w[lane][1] : 0;
#pragma unroll
        for (int o = 16; o >= 1; o >>= 1) {
            a += shfl_xor_u128(a, o);
            b += shfl_xor_u128(b, o);
        }
        if (lane != 0) return;
        DevMetrics *m = d.metrics;
        atomicAdd(&m->requests, (unsigned long long)n);
        atomicAdd(&m->prompt_tokens, (unsigned long long)t[0]);
        atomicAdd(&m->hit_tokens, (unsigned long long)t[1]);
        atomicAdd(&m->switched, (unsigned long long)t[2]);
        atomicAdd(&m->est_slo_met, (unsigned long long)t[3]);
        m->pend_n = t[4];
        m->pend_s1[0] = (uint64_t)a;
        m->pend_s1[1] = (uint64_t)(a >> 64);
        m->pend_s2[0] = (uint64_t)b;
        m->pend_s2[1] = (uint64_t)(b >> 64);
        m->pend = 1;
    }
}


// ---------------------------------------------------------------------------
// Choices in arrival order, pipelined over chunks of requests.
//
// What bounds a choice kernel is the chain of decisions that share an
// instance: on batches of hot templates about a third of the requests follow
// one another through the same pair.  So one warp does nothing but decide,
// and everything else is kept out of its way:
//   stage   a warp per window of 32 requests loads the requests and finds
//           which request of its window each one follows on each of its
//           candidates, and its level, one more than the largest of those.
//           Both depend on the candidates alone, so they are known before
//           any decision;
//   decide  warp 0, window by window, level by level.  Loads that fit 32 bits
//           pass from request to request (registers and shuffles for two
//           candidates, a shared-memory row per lane for d); every lane decides
//           at every level, so nothing waits or branches, and a request is
//           right from its level on.  Larger loads stay in shared memory: the
//           requests of one level share no instance, so reading W and writing
//           W[choice] for all of them at once equals arrival order exactly;
//   emit    a warp per window places the requests among their instances'
//           records and queue entries and writes every output.
// Chunk t is staged while chunk t - 1 is decided and chunk t - 2 emitted,
// over three staging buffers.  Measured (GB300, kernel time for 4,096 agent
// prompts, two and four candidates): 191 and 5,200 us with rounds found by
// votes and with one thread, 82 and 164 us so (84 and 200 cycles a level, 470
// a window).
constexpr uint8_t kNoLevel = 255;

// The deciding warp has its SM sub-partition to itself (warps are dealt to the
// four by their number): every fourth warp only meets the barriers.  Beside
// emitting or staging warps the same chain ran 10-20 % longer (a pass of 4,096
// agent prompts 250 and 230 us, min TTFT over 64 instances 680 and 615).
template <uint32_t kChunk, uint32_t kStageThreads = kChunk>
struct Pipe {
    static constexpr uint32_t kWorkers = (kChunk + kStageThreads) / 32;   // the emitting, then the staging warps
    static constexpr uint32_t kThreads = 32 * (1 + kWorkers + (kWorkers - 1) / 3);
};

// begin() by the deciding warp while the first chunk is staged; stage(buffer, k,
// m, base), decide(buffer, m), emit(buffer, k, m, base): k
// the thread's number among its role's (an emitting thread's request of the
// chunk; whole windows call, k >= m past the batch's end), m the chunk's
// requests, base its first request.
template <uint32_t kChunk, uint32_t kStageThreads, class BeginF, class StageF, class DecideF, class EmitF>
__device__ __forceinline__ void choice_pipeline(uint32_t n, BeginF begin, StageF stage, DecideF decide, EmitF emit) {
    const uint32_t nc = (n + kChunk - 1) / kChunk, wid = threadIdx.x >> 5;
    const uint32_t w = 32 * (wid - 1 - wid / 4) + (threadIdx.x & 31);   // number among the workers (wid % 4 != 0)
    for (uint32_t t = 0; t < nc + 2; ++t) {
        if (wid == 0) {
            if (t == 0) begin();
            else if (t <= nc) decide((t - 1) % 3, min(kChunk, n - (t - 1) * kChunk));
        } else if (wid % 4 == 0) {
        } else if (w < kChunk) {
            if (t >= 2) emit((t - 2) % 3, w, min(kChunk, n - (t - 2) * kChunk), (t - 2) * kChunk);
        } else if (w < kChunk + kStageThreads) {
            if (t < nc) stage(t % 3, w - kChunk, min(kChunk, n - t * kChunk), t * kChunk);
        }
        __syncthreads();
    }
}

// How the requests of a window follow one another: for each of this lane's ND
// candidates c (0xFFFFFFFF past the batch's end; distinct instances) the latest
// earlier request of the window that names the same instance, as from[f] =
// its lane * kStride + its candidate's number (kNone: none), and in the result
// bit f whether no later one does.  lev: the request's level, one more than
// the largest of those it follows (0: none); nlev: the window's number of
// levels.  Whole warp.
constexpr uint32_t kNone = 0xFFFFFFFFu;
template <uint32_t ND, uint32_t kStride>
__device__ __forceinline__ uint32_t window_links(const uint32_t (&c)[ND], bool valid, int lane, uint32_t (&from)[ND],
                                                 uint32_t &lev, uint32_t &nlev) {
    uint32_t later = 0;
#pragma unroll
    for (uint32_t f = 0; f < ND; ++f) from[f] = kNone;
    const int held = __popc(__ballot_sync(0xffffffffu, valid));   // the valid lanes are the first ones
#pragma unroll 4
    for (int j = 0; j < held; ++j) {
        const bool before = j < lane, after = j > lane;
#pragma unroll
        for (uint32_t y = 0; y < ND; ++y) {
            const uint32_t o = __shfl_sync(0xffffffffu, c[y], j);
#pragma unroll
            for (uint32_t f = 0; f < ND; ++f) {
                from[f] = o == c[f] && before ? j * kStride + y : from[f];
                later |= o == c[f] && after ? 1u << f : 0u;
            }
        }
    }
    lev = 0;
    for (bool more = true; more;) {
        uint32_t nl = 0;
#pragma unroll
        for (uint32_t f = 0; f < ND; ++f) {
            const uint32_t x = __shfl_sync(0xffffffffu, lev, from[f] / kStride);   // (kNone: any lane)
            nl = max(nl, valid && from[f] != kNone ? x + 1 : 0);
        }
        more = __any_sync(0xffffffffu, nl != lev);
        lev = nl;
    }
    nlev = __reduce_max_sync(0xffffffffu, valid ? lev + 1 : 0);
    return valid ? ~later & ((1u << ND) - 1u) : 0;
}

// Each request is staged as (a, b): a = the candidate with more cached
// blocks (c1 on equal hits), u = uncached work on each, and
// thr = SLO - u_a (-1 when u_a alone exceeds the SLO or the hits are equal),
// so the rule of Sec. 3.2 becomes: choose b iff W_b < W_a and W_a > thr
// (ttft_a = W_a + u_a > SLO); the SLO switch fired iff hits differ and
// W_a > thr.  The pair variants use the general form: choose b iff
// W_a > thr and (k_b < k_a or (k_b == k_a and tieb)), with k = W (+ u when
// the rule compares TTFTs) and tieb set where a tie goes to b (= c1).
constexpr uint32_t kChoiceChunk = 256;
constexpr uint64_t kSmall = 1ull << 30;   // loads below it are decided in 32 bits
constexpr uint32_t kWorkShift = 10;
constexpr uint64_t kWorkUnit = (1ull << kWorkShift) - 1;
struct ChoiceStage {
    uint64_t ua[kChoiceChunk], ub[kChoiceChunk];
    int64_t thr[kChoiceChunk];
    uint64_t Wa[kChoiceChunk], Wb[kChoiceChunk];
    uint32_t ab[kChoiceChunk];     // a | b << 14 | (a is c2) << 28 | (hits differ) << 29 | tieb << 30 | addu << 31
    // the same for a decision in 32 bits: a | b << 16, link, low words of ua and ub; thr (INT32_MAX at most) and lead
    // (pair rules: choose b iff W_b - W_a < lead and W_a > thr)
    uint4 rec[kChoiceChunk];
    int2 lim[kChoiceChunk];
    uint4 req[kChoiceChunk];       // the request's length, blocks and hit tokens on c1 and c2
    uint32_t wsum[kChoiceChunk / 32];   // per window: sum of the larger of both works, in units of 2^kWorkShift (rounded up)
    uint32_t nlev[kChoiceChunk / 32];
    uint8_t lev[kChoiceChunk], pickb[kChoiceChunk];
};

// link: bits 0-4 the lane that the request follows on a, bit 5 set: as that
// lane's b, bit 6: there is one, bit 7: no later request of the window names a;
// bits 8-15 the same for b; from bit 16 on the window's number of levels.

// W and PT (8 bytes each) per instance, then the staging buffers.
size_t choice_smem(uint32_t M) { return size_t(M) * 16 + 3 * sizeof(ChoiceStage); }

// kPairRules: the general form (the pair variants and global cache
// affinity); false compiles DualMap's rule alone.
//
// Bound: about 1,250 dependent levels on an agent batch (4,096 requests, 64
// instances, 200 templates).
template <bool kPairRules>
__global__ void __launch_bounds__(Pipe<kChoiceChunk>::kThreads, 1) k_choice(DevState d, dm_route_out o, uint32_t n,
                                                                         uint64_t seq0, uint64_t t_batch) {
    pdl_enter();
    extern __shared__ __align__(16) unsigned char smem[];
    if (has_err(d.err)) return;
    if (blockIdx.x > 0) {   // beside the choice: the segment carries the commit needs
        carries_role(d, o, n, blockIdx.x - 1, gridDim.x - 1);
        return;
    }
    uint64_t *W = reinterpret_cast<uint64_t *>(smem);
    uint64_t *PT = W + d.M;
    ChoiceStage *const SB = reinterpret_cast<ChoiceStage *>(PT + d.M);
    const int lane = threadIdx.x & 31;
    uint32_t live_bits = 0;   // bit k: instance threadIdx.x + k * blockDim.x is live (M <= 16 * 704)
    for (uint32_t i = threadIdx.x, k = 0; i < d.M; i += blockDim.x, ++k) {
        W[i] = d.W[i];
        PT[i] = d.q_tail[i];
        live_bits |= uint32_t(d.inst_state[i] == 1) << k;
    }
    const uint64_t cost = d.cost, slo = d.slo;
    const uint32_t rule = kPairRules ? d.rule : uint32_t(DM_RULE_DUALMAP);
    MetricSums ms{0, 0, 0, 0};

    auto stage = [&](uint32_t buf, uint32_t k, uint32_t m, uint32_t base) {
        if ((k & ~31u) >= m) return;   // no request in this window
        ChoiceStage &S = SB[buf];
        const bool valid = k < m;
        uint32_t ids[2] = {kNone, kNone}, u32[2] = {0, 0};
        uint64_t most = 0;
        if (valid) {
            const uint32_t r = base + k;
            const uint32_t L = d.r_L[r], nblk = d.r_nblk[r];
            const uint32_t h1 = hit_tokens(d.r_m1[r], nblk, d.B), h2 = hit_tokens(d.r_m2[r], nblk, d.B);
            const uint32_t c1 = d.r_c1[r], c2 = d.r_c2[r];
            // global cache affinity always takes c1: orient it as a, never b
            S.req[k] = make_uint4(L, nblk, h1, h2);
            const bool a2 = rule != DM_RULE_CACHE_AFFINITY && h2 > h1;
            const bool differ = h1 != h2;
            const uint64_t ua = cost * (L - (a2 ? h2 : h1)), ub = cost * (L - (a2 ? h1 : h2));
            constexpr int64_t kNever = INT64_MAX;   // W_a never exceeds it: keep a
            int64_t thr = -1;
            bool tieb = false, addu = false;
            const bool affine = rule == DM_RULE_PAIR_CACHE_AFFINITY ||
                                (rule == DM_RULE_PAIR_PREBLE && 2ull * max(h1, h2) > L);
            if (rule == DM_RULE_DUALMAP) {
                thr = (!differ || ua > slo) ? -1 : (int64_t)min(slo - ua, (uint64_t)kNever);
            } else if (rule == DM_RULE_CACHE_AFFINITY) {
                thr = kNever;
            } else if (affine) {
                thr = differ ? kNever : -1;
            } else {                       // least loaded / min TTFT (and Preble below half)
                tieb = a2;
                addu = rule != DM_RULE_PAIR_LEAST_LOADED;
            }
            S.ua[k] = ua;
            S.ub[k] = ub;
            S.thr[k] = thr;
            S.ab[k] = (a2 ? c2 : c1) | ((a2 ? c1 : c2) << 14) | (uint32_t(a2) << 28) | (uint32_t(differ) << 29) |
                      (uint32_t(tieb) << 30) | (uint32_t(addu) << 31);
            ids[0] = a2 ? c2 : c1;
            ids[1] = a2 ? c1 : c2;
            u32[0] = (uint32_t)ua;
            u32[1] = (uint32_t)ub;
            S.lim[k] = make_int2((int32_t)min(thr, (int64_t)INT32_MAX),
                                 (addu ? (int32_t)(u32[0] - u32[1]) : 0) + (tieb ? 1 : 0));
            most = min(max(ua, ub), kSmall);
        }
        uint32_t lev, nlev, from[2];
        const uint32_t last = window_links<2, 2>(ids, valid, lane, from, lev, nlev);
        uint32_t link = nlev << 16;
#pragma unroll
        for (uint32_t f = 0; f < 2; ++f) {
            const uint32_t x = valid && from[f] != kNone ? from[f] / 2 | (from[f] & 1u) << 5 | 1u << 6 : 0;
            link |= (x | ((last >> f) & 1u) << 7) << (8 * f);
        }
        S.rec[k] = make_uint4(valid ? ids[0] | ids[1] << 16 : 0, link, u32[0], u32[1]);
        S.lev[k] = valid ? (uint8_t)lev : kNoLevel;
        const uint32_t sum = __reduce_add_sync(0xffffffffu, (uint32_t)((most + kWorkUnit) >> kWorkShift));
        if (lane == 0) {
            S.nlev[k / 32] = nlev;
            S.wsum[k / 32] = sum;
        }
    };

    // one chunk whose loads stay below 2^30.  Every lane decides its request at
    // every level, from the loads that the requests it follows leave (the
    // loads at the window's start where there is none), so a request is right
    // from its level on and the whole window after nlev levels: no lane waits
    // or branches.  A level is four shuffles and a dozen operations in
    // registers.  The window's last request on an instance leaves its load in
    // W; the next window's staged values are read meanwhile.
    uint64_t bound = 0;   // no load exceeds it, unless it is kSmall
    auto begin = [&] {
        for (uint32_t i = lane; i < d.M; i += 32) bound = max(bound, min(d.W[i], kSmall));
        bound = __reduce_max_sync(0xffffffffu, (uint32_t)bound);
    };
    auto decide32 = [&](ChoiceStage &S, uint32_t m) {
        volatile uint32_t *const W32 = reinterpret_cast<volatile uint32_t *>(W);   // low words; the high ones are 0
        uint4 nr = S.rec[lane];
        int2 nl = S.lim[lane];   // past the batch's end: unused
        for (uint32_t w0 = 0; w0 < m; w0 += 32) {
            const uint4 x = nr;
            const int32_t thr = nl.x, lead = kPairRules ? nl.y : 0;
            const uint32_t a = x.x & 0xFFFF, b = x.x >> 16, link = x.y;
            const uint32_t nlev = __reduce_max_sync(0xffffffffu, link >> 16);   // uniform: the loop below has no divergence
            uint32_t A = W32[2 * a], B = W32[2 * b];
            const uint32_t kn = (w0 + 32 < m ? w0 + 32 : 0) + lane;
            nr = S.rec[kn];
            nl = S.lim[kn];
            const int sa = link & 31, sb = (link >> 8) & 31;
            // where A and B come from: that lane's a, that lane's b, or here
            auto mask = [&](uint32_t bits, uint32_t is) { return (bits & 0x60u) == is ? ~0u : 0u; };
            const uint32_t ma0 = mask(link, 0x40u), ma1 = mask(link, 0x60u);
            const uint32_t mb0 = mask(link >> 8, 0x40u), mb1 = mask(link >> 8, 0x60u);
            const uint32_t Ah = A & ~(ma0 | ma1), Bh = B & ~(mb0 | mb1);
            int32_t pb;   // all ones: b
            uint32_t oA, oB;
            auto step = [&] {
                pb = ((int32_t)(B - A - lead) & (thr - (int32_t)A)) >> 31;
                oA = A + (x.z & ~pb);
                oB = B + (x.w & pb);
            };
            auto level = [&] {
                const uint32_t A0 = __shfl_sync(0xffffffffu, oA, sa), A1 = __shfl_sync(0xffffffffu, oB, sa);
                const uint32_t B0 = __shfl_sync(0xffffffffu, oA, sb), B1 = __shfl_sync(0xffffffffu, oB, sb);
                A = (A0 & ma0) | Ah | (A1 & ma1);
                B = (B0 & mb0) | Bh | (B1 & mb1);
                step();
            };
            step();
#pragma unroll 1
            for (uint32_t l = 1; l < nlev; l += 2) {   // a level more than there are changes nothing
                level();
                level();
            }
            if (link & 0x80u) W32[2 * a] = oA;
            if (link & 0x8000u) W32[2 * b] = oB;
            __syncwarp();
            const uint32_t k = w0 + lane;
            S.Wa[k] = A;
            S.Wb[k] = B;
            S.pickb[k] = pb != 0;
        }
    };

    auto decide = [&](uint32_t buf, uint32_t m) {
        ChoiceStage &S = SB[buf];
        bound = min(bound + (uint64_t(__reduce_add_sync(0xffffffffu, (uint32_t)lane < (m + 31) / 32 ? S.wsum[lane] : 0))
                             << kWorkShift),
                    kSmall);
        if (bound < kSmall) {
            decide32(S, m);
            return;
        }
        volatile uint64_t *const Wv = W;
        for (uint32_t w0 = 0; w0 < m; w0 += 32) {
            const uint32_t k = w0 + lane;
            const uint32_t mine = S.lev[k], nlev = S.nlev[w0 / 32];
            const uint32_t ab = mine != kNoLevel ? S.ab[k] : 0;
            const uint32_t a = ab & 0x3FFF, b = (ab >> 14) & 0x3FFF;
            const uint64_t ua = S.ua[k], ub = S.ub[k];   // past the batch's end: unused
            const int64_t thr = S.thr[k];
            const bool tieb = (ab >> 30) & 1u;
            const uint64_t xa = (ab >> 31) ? ua : 0, xb = (ab >> 31) ? ub : 0;
            uint64_t oWa = 0, oWb = 0;
            bool opb = false;
            for (uint32_t l = 0; l < nlev; ++l) {
                const uint64_t Wa = Wv[a], Wb = Wv[b];
                bool pb;
                if constexpr (kPairRules) {
                    const uint64_t ka = Wa + xa, kb = Wb + xb;
                    pb = (int64_t)Wa > thr && (kb < ka || (kb == ka && tieb));
                } else {
                    pb = Wb < Wa && (int64_t)Wa > thr;
                }
                const uint64_t na = Wa + ua, nb = Wb + ub;
                if (mine == l) {
                    Wv[pb ? b : a] = pb ? nb : na;
                    oWa = Wa;
                    oWb = Wb;
                    opb = pb;
                }
                __syncwarp();
            }
            S.Wa[k] = oWa;
            S.Wb[k] = oWb;
            S.pickb[k] = opb;
        }
    };

    auto emit = [&](uint32_t buf, uint32_t k, uint32_t m, uint32_t base) {
        const ChoiceStage &S = SB[buf];
        const bool valid = k < m;
        const uint32_t r = base + k;
        const uint32_t ab = valid ? S.ab[k] : 0;
        const uint32_t a = ab & 0x3FFF, b = (ab >> 14) & 0x3FFF;
        const bool a_is_c2 = (ab >> 28) & 1, differ = (ab >> 29) & 1;
        const bool pb = valid && S.pickb[k];
        const uint32_t ch = pb ? b : a;
        const uint4 rq = valid ? S.req[k] : make_uint4(0, 0, 0, 0);
        const uint32_t L = rq.x, nbr = rq.y, h1 = rq.z, h2 = rq.w;
        const uint32_t qh = d.q_head[ch];   // (a = 0 past the batch's end)
        const uint64_t pt = record_place<kChoiceChunk>(PT, ch, (uint64_t(nbr) << 32) + 1, valid, k / 32,
                                                       (m + 31) / 32, lane);
        if (!valid) return;
        const uint64_t ta = S.Wa[k] + S.ua[k], tb = S.Wb[k] + S.ub[k];
        o.ttft1[r] = a_is_c2 ? tb : ta;
        o.ttft2[r] = a_is_c2 ? ta : tb;
        const bool sw = differ && (rule == DM_RULE_DUALMAP ? (int64_t)S.Wa[k] > S.thr[k] : pb);
        o.chosen[r] = ch;
        o.switched[r] = sw;
        d.r_final[r] = ch;
        ms.tokens += L;
        ms.hits += (ch == (a_is_c2 ? b : a)) ? h1 : h2;
        ms.sw += sw;
        ms.est += (pb ? tb : ta) <= slo;
        if (ta > slo && tb > slo) d.info->both_over = 1;
        d.r_touchoff[r] = pt >> 32;          // offset among this batch's records of ch
        const uint32_t slot = (uint32_t)pt;
        if (slot - qh >= d.Q) {
            set_err(d.err, DM_ERR_CAPACITY);
            return;
        }
        QEntry e;
        e.seq = seq0 + r;
        e.work = e.remaining = pb ? S.ub[k] : S.ua[k];
        e.L = L;
        e.c1 = a_is_c2 ? b : a;
        e.c2 = a_is_c2 ? a : b;
        e.h1 = h1;
        e.h2 = h2;
        e.moved = 0;
        e.arrival = t_batch;
        // its keys' ring position: the instance's ring tail at the batch's
        // start plus this batch's earlier blocks queued there (the same
        // order as its touch records)
        e.koff = d.KQ ? d.kr_tail[ch] + (pt >> 32) : 0;
        if (d.KQ) d.r_koff[r] = e.koff;
        DM_CHECK(ch < d.M, d.err);
        d.q[uint64_t(ch) * d.Q + (slot & (d.Q - 1))] = e;
    };

    // (W and PT are first read after the first chunk's barrier)
    choice_pipeline<kChoiceChunk, kChoiceChunk>(n, begin, stage, decide, emit);
    unsigned __int128 S1 = 0, S2 = 0;
    uint32_t cnt = 0;
    for (uint32_t i = threadIdx.x, k = 0; i < d.M; i += blockDim.x, ++k) {
        d.W[i] = W[i];
        d.q_tail[i] = (uint32_t)PT[i];
        d.log_adv[i] = PT[i] >> 32;
        if (d.KQ) {   // the batch's keys on instance i take its ring's next positions
            const uint64_t nt = d.kr_tail[i] + (PT[i] >> 32);
            if (nt - d.kr_head[i] > d.KQ) set_err(d.err, DM_ERR_CAPACITY);
            d.kr_tail[i] = nt;
        }
        if ((live_bits >> k) & 1u) {
            S1 += W[i];
            S2 += (unsigned __int128)W[i] * W[i];
            ++cnt;
        }
    }
    if (threadIdx.x == 0) d.info->final_dirty = 0;
    finish_metrics(d, n, ms, S1, S2, cnt);
}

// ---------------------------------------------------------------------------
// Cluster-wide rules.

// Hit tokens of every request on every live instance (0 elsewhere), against
// the index as of the start of the batch: a warp per request and 32
// instances, a lane per instance.  The keys resident on an instance are
// closed under prefixes (see the routing kernel), so a lane tests block 0
// and, where that is resident (most instances miss it), finds the run's end:
// first whether it is the longer of the runs on the request's two candidates
// (a shared prefix that is resident on several instances mostly ends at the
// same block), then by three probes a round, each round leaving a quarter of
// the range; lanes that probe the same block read the same prefix value.
// Bound by dependent 16-byte index reads.  4,096 agent prompts x 64
// instances, GB300: 822 us with a warp per pair that walked the run, 90 us so.
constexpr int kAllBlock = 256;

// resident_at past the home slot (not inlined: three of these in a round).
static __device__ __noinline__ bool resident_past_home(const Slot *t, uint64_t mask, uint64_t key, uint64_t home,
                                                       uint64_t front, uint32_t *err, uint64_t loop_limit) {
    return table_pos1(t, mask, key, home, err, loop_limit) > front;
}

__global__ void __launch_bounds__(kAllBlock, 4) k_probe_all(DevState d, uint32_t n) {
    pdl_enter();
    if (has_err(d.err)) return;
    const int lane = threadIdx.x & 31;
    const uint32_t groups = (d.M + 31) / 32;
    const uint64_t total = uint64_t(n) * groups, nw = uint64_t(gridDim.x) * (kAllBlock / 32);
    const uint64_t mask = d.S - 1;
    for (uint64_t p = (uint64_t(blockIdx.x) * kAllBlock + threadIdx.x) / 32; p < total; p += nw) {
        const uint32_t r = (uint32_t)(p / groups), i = (uint32_t)(p - uint64_t(r) * groups) * 32 + lane;
        if (i >= d.M) continue;
        uint32_t h = 0;
        if (d.inst_state[i] == 1) {
            const uint32_t nblk = d.r_nblk[r], s0 = d.r_segoff[r];
            const uint64_t *pl = d.plocal + d.r_blkoff[r];
            const Slot *t = d.table[i];
            const uint64_t front = d.log_front[i];
            // which of blocks b[0 .. 2] are resident
            auto resident = [&](const uint32_t (&b)[3], bool (&in)[3]) {
                uint64_t key[3], home[3];
                Slot sl[3];
#pragma unroll
                for (int q = 0; q < 3; ++q) {
                    const uint64_t carry = d.seg_carry[s0 + b[q] / kSegBlocks];
                    key[q] = cache_key(pl[b[q]] + carry, d.Sc);
                    home[q] = group_home(cache_key(pl[b[q] & ~(kGroup - 1)] + carry, d.Sc), b[q], mask);
                    sl[q] = load_slot(t + home[q]);
                }
#pragma unroll
                for (int q = 0; q < 3; ++q)
                    in[q] = sl[q].key == key[q] ? sl[q].pos1 > front
                                                : sl[q].key != 0 && resident_past_home(t, mask, key[q], home[q], front,
                                                                                       d.err, d.loop_limit);
            };
            const uint64_t key0 = cache_key(pl[0] + d.seg_carry[s0], d.Sc), home0 = group_home(key0, 0, mask);
            if (resident_at(t, mask, key0, home0, front, load_slot(t + home0), d.err, d.loop_limit)) {
                const uint32_t g = max(min(d.r_m1[r], nblk), min(d.r_m2[r], nblk));   // first miss on a candidate
                RunEnd end(nblk, g);
                while (end.open()) {
                    bool in[3];
                    resident(end.b, in);
                    end.narrow(in);
                }
                h = end.hi;
            }
        }
        d.h_all[uint64_t(r) * d.M + i] = h * d.B;
    }
}

// The same for few pairs of request and instance: a warp per pair tests the
// first blocks of 32 segments a round, then the segment that holds the run's
// end (the routing kernel's way), four or five round trips instead of a dozen.
// A pass of min TTFT over agent prompts and 64 instances, GB300, this way and a
// lane per pair: 1,024 pairs 53 and 59 us, 16,384 pairs 81 and 86, 32,768 pairs
// 115 and 107.
constexpr uint32_t kPairWarps = 16384;

__global__ void __launch_bounds__(kAllBlock) k_probe_pairs(DevState d, uint32_t n) {
    pdl_enter();
    if (has_err(d.err)) return;
    const int lane = threadIdx.x & 31;
    const uint32_t p = (blockIdx.x * kAllBlock + threadIdx.x) / 32;
    if (p >= n * d.M) return;
    const uint32_t r = p / d.M, i = p - r * d.M;
    uint32_t h = 0;
    if (d.inst_state[i] == 1) {
        const uint32_t nblk = d.r_nblk[r], s0 = d.r_segoff[r], nseg = (nblk + kSegBlocks - 1) / kSegBlocks;
        const uint64_t *pl = d.plocal + d.r_blkoff[r];
        const Slot *const t[1] = {d.table[i]};
        const uint64_t front[1] = {d.log_front[i]}, mask = d.S - 1;
        uint32_t js = nseg, run[1];   // first segment whose first block is missing
        for (uint32_t g0 = 0; g0 < nseg; g0 += 32) {
            const uint32_t sg = g0 + lane;
            const uint64_t key[1] = {
                sg < nseg ? cache_key(pl[uint64_t(sg) * kSegBlocks] + d.seg_carry[s0 + sg], d.Sc) : 0};
            const uint64_t home[1] = {group_home(key[0], 0, mask)};   // a segment's first block anchors its own group
            const int look[1][1] = {{sg < nseg ? look_at(load_slot(t[0] + home[0]), key[0], front[0]) : kOut}};
            leading_runs<1, 1>(look, t, front, mask, key, home, lane, d.err, d.loop_limit, run);
            if (run[0] < min(32u, nseg - g0)) {
                js = g0 + run[0];
                break;
            }
        }
        if (js) {
            const uint32_t c0 = (js - 1) * kSegBlocks, cn = min(kSegBlocks, nblk - c0);
            const uint64_t carry = d.seg_carry[s0 + js - 1];
            uint64_t key[2], home[2];
            Slot s[2];
            int look[1][2];
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                const uint32_t e = 32 * q + lane;
                key[q] = e < cn ? cache_key(pl[c0 + e] + carry, d.Sc) : 0;
                home[q] = group_home(group_anchor(key[q], lane), c0 + e, mask);
                s[q] = e < cn ? load_slot(t[0] + home[q]) : Slot{0, 0};
            }
#pragma unroll
            for (int q = 0; q < 2; ++q) look[0][q] = 32u * q + lane < cn ? look_at(s[q], key[q], front[0]) : kOut;
            leading_runs<1, 2>(look, t, front, mask, key, home, lane, d.err, d.loop_limit, run);
            h = run[0] < cn ? c0 + run[0] : min(js * kSegBlocks, nblk);
        }
    }
    if (lane == 0) d.h_all[uint64_t(r) * d.M + i] = h * d.B;
}

// ---------------------------------------------------------------------------
// The cluster-wide choice over up to 512 instances, pipelined like the pair
// choice.  Every request depends on the one before it, so the chain is the
// argmin over the instances and it alone is left to the deciding warp: the
// loads stay in its registers (lane l holds the live ids of list indices
// J l .. J l + J - 1), as 32-bit offsets from the smallest load, and one
// request is J compares, a 32-bit minimum over the warp, a vote, and an add in
// the winning lane, which stores the index it holds.  The lowest lane with the
// smallest key holds the lowest id.  A chunk whose loads and work do not fit
// 31 bits is decided in 64 bits instead.  The hits come into shared memory a
// chunk ahead; the loads that a request found on its candidates follow from
// the loads at the chunk's start and the choices before it, which the emitting
// warps add up.
// 4,096 agent prompts on 64 instances, min TTFT, GB300: 1,678 us with 64-bit
// keys and loads in shared memory, three reductions a request, and staging
// and emission between the chunks, 204 us so (100 cycles a request).
constexpr uint32_t kGlobalStageThreads = 256;
template <uint32_t J>
struct GlobalPipe {
    static constexpr uint32_t kChunk = J <= 8 ? 64 : 32;   // three buffers of hits fit at 512 instances
    static constexpr uint32_t kThreads = Pipe<kChunk, kGlobalStageThreads>::kThreads;
    struct Stage {
        alignas(16) uint32_t hit[kChunk][32 * J];
        uint64_t cl[kChunk];      // cost x L
        uint64_t w0[kChunk / 32][32 * J];   // loads at the start of each 32 requests
        uint64_t wk[kChunk];      // work that the request adds to the chosen instance
        uint32_t hmax[kChunk];    // 0xFFFFFFFF: no affinity
        uint32_t ch[kChunk];      // list index chosen
    };
    static size_t smem(uint32_t M) { return 32 * J * 20 + (size_t(M) * 2 + 15) / 16 * 16 + 3 * sizeof(Stage); }
};

template <uint32_t J>
__global__ void __launch_bounds__(GlobalPipe<J>::kThreads, 1) k_choice_all(DevState d, dm_route_out o, uint32_t n,
                                                                        uint64_t seq0, uint64_t t_batch) {
    pdl_enter();
    using P = GlobalPipe<J>;
    using Stage = typename P::Stage;
    constexpr uint32_t kN = 32 * J, kChunk = P::kChunk;
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ uint32_t s_wcnt[32];
    if (has_err(d.err)) return;
    // by list index: load, records << 32 | queue tail, id; by id: list index
    uint64_t *W = reinterpret_cast<uint64_t *>(smem), *PT = W + kN;
    uint32_t *live = reinterpret_cast<uint32_t *>(PT + kN);
    uint16_t *inv = reinterpret_cast<uint16_t *>(live + kN);
    Stage *const SB = reinterpret_cast<Stage *>(smem + kN * 20 + (size_t(d.M) * 2 + 15) / 16 * 16);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    uint32_t nl = 0;   // live ids in ascending order
    for (uint32_t base = 0; base < d.M; base += blockDim.x) {
        const uint32_t i = base + threadIdx.x;
        const bool f = i < d.M && d.inst_state[i] == 1;
        const uint32_t bal = __ballot_sync(0xffffffffu, f);
        if (lane == 0) s_wcnt[wid] = __popc(bal);
        __syncthreads();
        uint32_t off = nl, tot = 0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
            off += w < wid ? s_wcnt[w] : 0;
            tot += s_wcnt[w];
        }
        if (f) {
            const uint32_t k = off + __popc(bal & ((1u << lane) - 1));
            live[k] = i;
            inv[i] = (uint16_t)k;
            W[k] = d.W[i];
            PT[k] = d.q_tail[i];
        }
        nl += tot;
        __syncthreads();
    }
    if (nl == 0) {   // the host requires two
        if (threadIdx.x == 0) set_err(d.err, DM_ERR_NO_INSTANCES);
        return;
    }
    const uint64_t cost = d.cost, slo = d.slo;
    const uint32_t rule = d.rule;
    MetricSums ms{0, 0, 0, 0};

    auto stage = [&](uint32_t buf, uint32_t k, uint32_t m, uint32_t base) {
        Stage &S = SB[buf];
        constexpr uint32_t kWarps = kGlobalStageThreads / 32, G = 16 / J;   // a warp takes G requests' loads at a time
        for (uint32_t q = k >> 5; q < m; q += kWarps * G) {
            uint32_t h[G][J], L[G];
#pragma unroll
            for (uint32_t g = 0; g < G; ++g) {
                const uint32_t rr = q + g * kWarps;
                const uint32_t *ha = d.h_all + uint64_t(base + rr) * d.M;
                L[g] = rr < m ? d.r_L[base + rr] : 0;
#pragma unroll
                for (uint32_t j = 0; j < J; ++j) {
                    const uint32_t x = j * 32 + lane;
                    h[g][j] = rr < m && x < nl ? ha[live[x]] : 0;
                }
            }
#pragma unroll
            for (uint32_t g = 0; g < G; ++g) {
                const uint32_t rr = q + g * kWarps;
                if (rr >= m) break;
                uint32_t hmax = 0;
#pragma unroll
                for (uint32_t j = 0; j < J; ++j) {
                    S.hit[rr][j * 32 + lane] = h[g][j];
                    hmax = max(hmax, h[g][j]);
                }
                if (rule == DM_RULE_PREBLE) hmax = __reduce_max_sync(0xffffffffu, hmax);
                if (lane == 0) {
                    S.cl[rr] = cost * L[g];
                    S.hmax[rr] = rule == DM_RULE_PREBLE && 2ull * hmax > L[g] ? hmax : 0xFFFFFFFFu;
                }
            }
        }
    };

    // one chunk with loads (as offsets from lo) and work in 31 bits; w: this
    // lane's loads, moved on.  kPack: they leave room for the list index below
    // them, so the minimum over the warp is the choice itself; otherwise a vote
    // finds the lowest lane that holds the minimum.
    constexpr uint32_t kNever = 0x80000000u;
    constexpr uint32_t kIndexBits = J == 2 ? 6 : J == 4 ? 7 : J == 8 ? 8 : 9;
    auto decide32 = [&](auto kind, auto pack, Stage &S, uint32_t m, uint32_t (&w)[J], uint64_t lo) {
        constexpr uint32_t kRule = decltype(kind)::value;
        constexpr bool kPack = decltype(pack)::value;
        constexpr uint32_t kShift = kPack ? kIndexBits : 0;
        struct alignas(J >= 4 ? 16 : 8) Hits {
            uint32_t v[J];
        };
        const uint32_t c32 = (uint32_t)cost << kShift;
        if constexpr (kPack) {
#pragma unroll
            for (uint32_t j = 0; j < J; ++j)   // past the list: above every key that may win
                w[j] = w[j] == kNever ? kNever : w[j] << kShift | (lane * J + j);
        }
        // the next request's staged values, read while this one is decided
        Hits h = *reinterpret_cast<const Hits *>(&S.hit[0][lane * J]);
        uint32_t cl = (uint32_t)S.cl[0] << kShift, hm = S.hmax[0];
        for (uint32_t rr = 0; rr < m; ++rr) {
            if ((rr & 31u) == 0) {
#pragma unroll
                for (uint32_t j = 0; j < J; ++j)
                    if (lane * J + j < nl) S.w0[rr / 32][lane * J + j] = lo + (w[j] >> kShift);
            }
            uint32_t u[J], key[J];   // its work on each instance; its keys
#pragma unroll
            for (uint32_t j = 0; j < J; ++j) {
                u[j] = cl - c32 * h.v[j];
                const bool affine = kRule == DM_RULE_PREBLE && hm != 0xFFFFFFFFu;
                key[j] = w[j] + (kRule == DM_RULE_LEAST_LOADED || affine ? 0u : u[j]);
                if (affine && h.v[j] != hm) key[j] = 0xFFFFFFFFu;   // left out
            }
            const uint32_t nx = min(rr + 1, m - 1);
            h = *reinterpret_cast<const Hits *>(&S.hit[nx][lane * J]);
            cl = (uint32_t)S.cl[nx] << kShift;
            hm = S.hmax[nx];
            if constexpr (kPack) {
                uint32_t best = key[0];
#pragma unroll
                for (uint32_t j = 1; j < J; ++j) best = min(best, key[j]);
                best = __reduce_min_sync(0xffffffffu, best);
#pragma unroll
                for (uint32_t j = 0; j < J; ++j) w[j] += key[j] == best ? u[j] : 0u;   // keys differ in their index
                // (least loaded, affinity: the key is the load and its index; else the work lies above the index)
                if (lane == 0) S.ch[rr] = best & ((1u << kIndexBits) - 1u);
            } else {
                uint32_t bj[J];
#pragma unroll
                for (uint32_t j = 0; j < J; ++j) bj[j] = j;
#pragma unroll
                for (uint32_t s = 1; s < J; s *= 2)   // ties: the lower index
#pragma unroll
                    for (uint32_t j = 0; j + s < J; j += 2 * s) {
                        const bool less = key[j + s] < key[j];
                        key[j] = less ? key[j + s] : key[j];
                        bj[j] = less ? bj[j + s] : bj[j];
                    }
                const uint32_t kmin = __reduce_min_sync(0xffffffffu, key[0]);
                const uint32_t eq = __ballot_sync(0xffffffffu, key[0] == kmin);
                const uint32_t won = eq & (0u - eq) & (1u << lane) ? bj[0] : J;   // the lowest lane's index
#pragma unroll
                for (uint32_t j = 0; j < J; ++j) w[j] += won == j ? u[j] : 0u;
                if (won < J) S.ch[rr] = lane * J + won;
            }
        }
#pragma unroll
        for (uint32_t j = 0; j < J; ++j)
            if (lane * J + j < nl) W[lane * J + j] = lo + (w[j] >> kShift);
    };

    auto decide = [&](uint32_t buf, uint32_t m) {
        Stage &S = SB[buf];
        volatile uint64_t *const Wv = W;
        uint64_t w64[J], lo = ~0ull, hi = 0, work = 0;
        bool small = true;   // cost x L of every request fits 31 bits
#pragma unroll
        for (uint32_t j = 0; j < J; ++j) {
            const uint32_t x = lane * J + j;
            w64[j] = x < nl ? W[x] : ~0ull;
            if (x < nl) {
                lo = min(lo, w64[j]);
                hi = max(hi, w64[j]);
            }
        }
        for (uint32_t rr = lane; rr < m; rr += 32) {
            small &= S.cl[rr] < (1ull << 31);
            work += S.cl[rr];
        }
#pragma unroll
        for (int x = 16; x >= 1; x >>= 1) {
            lo = min(lo, shfl_xor_u64(lo, x));
            hi = max(hi, shfl_xor_u64(hi, x));
            work += shfl_xor_u64(work, x);
        }
        small = __all_sync(0xffffffffu, small);
        if (small && hi - lo < kNever && work < kNever - (hi - lo)) {
            uint32_t w[J];   // past the list: above every key that may win
#pragma unroll
            for (uint32_t j = 0; j < J; ++j) w[j] = lane * J + j < nl ? (uint32_t)(w64[j] - lo) : kNever;
            auto by_rule = [&](auto pack) {
                if (rule == DM_RULE_MIN_TTFT)
                    decide32(std::integral_constant<uint32_t, DM_RULE_MIN_TTFT>{}, pack, S, m, w, lo);
                else if (rule == DM_RULE_LEAST_LOADED)
                    decide32(std::integral_constant<uint32_t, DM_RULE_LEAST_LOADED>{}, pack, S, m, w, lo);
                else decide32(std::integral_constant<uint32_t, DM_RULE_PREBLE>{}, pack, S, m, w, lo);
            };
            if (hi - lo + work < (kNever >> kIndexBits)) by_rule(std::true_type{});
            else by_rule(std::false_type{});
        } else {
            for (uint32_t rr = 0; rr < m; ++rr) {
                if ((rr & 31u) == 0)
                    for (uint32_t x = lane; x < nl; x += 32) S.w0[rr / 32][x] = Wv[x];
                const uint64_t cl = S.cl[rr];
                const uint32_t hm = S.hmax[rr];
                // smallest (key, list index): three 32-bit reductions give the exact pair
                uint64_t bk = ~0ull;
                uint32_t bx = 0xFFFFFFFFu;
                for (uint32_t x = lane; x < nl; x += 32) {
                    const uint32_t h = S.hit[rr][x];
                    const uint64_t w = Wv[x];
                    const uint64_t key = rule == DM_RULE_LEAST_LOADED ? w
                                         : hm == 0xFFFFFFFFu          ? w + cl - cost * h
                                         : h == hm                    ? w
                                                                      : ~0ull;
                    if (key < bk || bx == 0xFFFFFFFFu) {
                        bk = key;
                        bx = x;
                    }
                }
                const uint32_t khi = __reduce_min_sync(0xffffffffu, (uint32_t)(bk >> 32));
                const uint32_t klo =
                    __reduce_min_sync(0xffffffffu, (uint32_t)(bk >> 32) == khi ? (uint32_t)bk : 0xFFFFFFFFu);
                const uint32_t x =
                    __reduce_min_sync(0xffffffffu, bk == ((uint64_t(khi) << 32) | klo) ? bx : 0xFFFFFFFFu);
                __syncwarp();
                if (lane == 0) {
                    Wv[x] = Wv[x] + cl - cost * S.hit[rr][x];
                    S.ch[rr] = x;
                }
                __syncwarp();
            }
        }
    };

    auto emit = [&](uint32_t buf, uint32_t k, uint32_t m, uint32_t base) {
        Stage &S = SB[buf];
        const bool valid = k < m;
        const uint32_t r = base + k, x = valid ? S.ch[k] : 0;
        const uint32_t nbr = valid ? d.r_nblk[r] : 0, h = valid ? S.hit[k][x] : 0;
        const uint64_t wk = valid ? S.cl[k] - cost * h : 0;
        if (valid) S.wk[k] = wk;
        const uint32_t L = valid ? d.r_L[r] : 0, c1 = valid ? d.r_c1[r] : 0, c2 = valid ? d.r_c2[r] : 0;
        const uint32_t f1 = valid ? d.r_m1[r] : 0, f2 = valid ? d.r_m2[r] : 0;
        const uint32_t ch = valid ? live[x] : live[0], qh = d.q_head[ch];
        // (its barriers also order the chunk's wk before the sums below)
        const uint64_t pt =
            record_place<kChunk>(PT, x, (uint64_t(nbr) << 32) + 1, valid, k / 32, (m + 31) / 32, lane);
        if (!valid) return;
        const uint32_t h1 = hit_tokens(f1, nbr, d.B), h2 = hit_tokens(f2, nbr, d.B);
        // the loads as the request found them
        const uint32_t x1 = inv[c1], x2 = inv[c2], q0 = k & ~31u;
        uint64_t wc = S.w0[q0 / 32][x], w1 = S.w0[q0 / 32][x1], w2 = S.w0[q0 / 32][x2];
        for (uint32_t q = q0; q < k; ++q) {
            const uint32_t cq = S.ch[q];
            const uint64_t wq = S.wk[q];
            wc += cq == x ? wq : 0;
            w1 += cq == x1 ? wq : 0;
            w2 += cq == x2 ? wq : 0;
        }
        const uint64_t t1 = w1 + cost * (L - h1), t2 = w2 + cost * (L - h2);
        o.ttft1[r] = t1;
        o.ttft2[r] = t2;
        o.chosen[r] = ch;
        o.switched[r] = 0;
        d.r_final[r] = ch;
        d.r_touchoff[r] = pt >> 32;
        ms.tokens += L;
        ms.hits += h;
        ms.est += wc + wk <= slo;
        if (t1 > slo && t2 > slo) d.info->both_over = 1;
        const uint32_t slot = (uint32_t)pt;
        if (slot - qh >= d.Q) {
            set_err(d.err, DM_ERR_CAPACITY);
            return;
        }
        QEntry e;
        e.seq = seq0 + r;
        e.work = e.remaining = wk;
        e.L = L;
        e.c1 = c1;
        e.c2 = c2;
        e.h1 = h1;
        e.h2 = h2;
        e.moved = 0;
        e.arrival = t_batch;
        e.koff = 0;
        DM_CHECK(ch < d.M, d.err);
        d.q[uint64_t(ch) * d.Q + (slot & (d.Q - 1))] = e;
    };

    choice_pipeline<kChunk, kGlobalStageThreads>(n, [] {}, stage, decide, emit);
    unsigned __int128 S1 = 0, S2 = 0;
    uint32_t cnt = 0;
    for (uint32_t i = threadIdx.x; i < d.M; i += blockDim.x) {
        if (d.inst_state[i] != 1) {
            d.log_adv[i] = 0;
            continue;
        }
        const uint32_t x = inv[i];
        d.W[i] = W[x];
        d.q_tail[i] = (uint32_t)PT[x];
        d.log_adv[i] = PT[x] >> 32;
        S1 += W[x];
        S2 += (unsigned __int128)W[x] * W[x];
        ++cnt;
    }
    if (threadIdx.x == 0) d.info->final_dirty = 0;
    finish_metrics(d, n, ms, S1, S2, cnt);
}

template <uint32_t J>
static cudaError_t launch_choice_all(const DevState &d, const dm_route_out &o, uint32_t n, uint64_t seq0,
                                     uint64_t t_batch, cudaStream_t st) {
    const size_t smem = GlobalPipe<J>::smem(d.M);
    static SmemOptIn opt;
    DM_TRY(opt_in_smem(opt, smem, k_choice_all<J>));
    return launch_pdl(k_choice_all<J>, 1, GlobalPipe<J>::kThreads, smem, st, d, o, n, seq0, t_batch);
}

// The same over any number of instances (max_instances above 512, where a
// lane could not keep its instances' loads in registers nor the chunks'
// hits fit three buffers).  k_choice_global: W and PT per instance and the
// live ids, then, for a chunk of `cap` requests, their per-request fields, their decisions and
// their hits on every live instance; cap is what the shared memory holds
// (at most 1024).  The decisions are written out in parallel after each
// chunk's sequential pass, which touches shared memory only.
__host__ __device__ inline size_t global_stage_off(uint32_t M) { return (size_t(M) * 20 + 15) / 16 * 16; }
constexpr uint32_t kGlobalReqBytes = 64;   // per-request fields and decision
constexpr uint32_t kGlobalReqMax = 1024;

__global__ void __launch_bounds__(1024) k_choice_global(DevState d, dm_route_out o, uint32_t n, uint64_t seq0,
                                                        uint64_t t_batch, uint32_t smem_bytes) {
    pdl_enter();
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ uint32_t s_wcnt[32];
    if (has_err(d.err)) return;
    uint64_t *W = reinterpret_cast<uint64_t *>(smem);
    uint64_t *PT = W + d.M;
    uint32_t *live = reinterpret_cast<uint32_t *>(PT + d.M);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    // live ids in ascending order
    uint32_t nl = 0;
    for (uint32_t base = 0; base < d.M; base += blockDim.x) {
        const uint32_t i = base + threadIdx.x;
        const bool f = i < d.M && d.inst_state[i] == 1;
        if (i < d.M) {
            W[i] = d.W[i];
            PT[i] = d.q_tail[i];
        }
        const uint32_t bal = __ballot_sync(0xffffffffu, f);
        if (lane == 0) s_wcnt[wid] = __popc(bal);
        __syncthreads();
        uint32_t off = nl;
        for (int w = 0; w < wid; ++w) off += s_wcnt[w];
        if (f) live[off + __popc(bal & ((1u << lane) - 1))] = i;
        uint32_t tot = 0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) tot += s_wcnt[w];
        nl += tot;
        __syncthreads();
    }
    const size_t off = global_stage_off(d.M);
    const uint64_t fit = (smem_bytes - off) / (kGlobalReqBytes + 4ull * max(nl, 1u));
    const uint32_t cap = fit < kGlobalReqMax ? (uint32_t)fit : kGlobalReqMax;
    uint64_t *s_pold = reinterpret_cast<uint64_t *>(smem + off);
    uint64_t *s_t1 = s_pold + cap, *s_t2 = s_t1 + cap, *s_wa = s_t2 + cap;
    uint32_t *s_L = reinterpret_cast<uint32_t *>(s_wa + cap);
    uint32_t *s_nb = s_L + cap, *s_c1 = s_nb + cap, *s_c2 = s_c1 + cap, *s_h1 = s_c2 + cap, *s_h2 = s_h1 + cap;
    uint32_t *s_ch = s_h2 + cap, *s_hch = s_ch + cap, *s_hits = s_hch + cap;
    const uint64_t cost = d.cost, slo = d.slo;
    const uint32_t rule = d.rule;
    MetricSums ms{0, 0, 0, 0};
    for (uint32_t r0 = 0; cap > 0 && r0 < n; r0 += cap) {
        const uint32_t m = min(cap, n - r0);
        __syncthreads();
        for (uint32_t x = threadIdx.x; x < m * nl; x += blockDim.x) {
            const uint32_t rr = x / nl, k = x - rr * nl;
            s_hits[x] = d.h_all[uint64_t(r0 + rr) * d.M + live[k]];
        }
        for (uint32_t rr = threadIdx.x; rr < m; rr += blockDim.x) {
            const uint32_t r = r0 + rr;
            s_L[rr] = d.r_L[r];
            s_nb[rr] = d.r_nblk[r];
            s_c1[rr] = d.r_c1[r];
            s_c2[rr] = d.r_c2[r];
            s_h1[rr] = hit_tokens(d.r_m1[r], s_nb[rr], d.B);
            s_h2[rr] = hit_tokens(d.r_m2[r], s_nb[rr], d.B);
        }
        __syncthreads();
        if (wid == 0) {
            for (uint32_t rr = 0; rr < m; ++rr) {
                const uint32_t L = s_L[rr];
                const uint32_t *hr = s_hits + rr * nl;
                bool affine = false;
                uint32_t hmax = 0;
                if (rule == DM_RULE_PREBLE) {
                    for (uint32_t k = lane; k < nl; k += 32) hmax = max(hmax, hr[k]);
                    hmax = __reduce_max_sync(0xffffffffu, hmax);
                    affine = 2ull * hmax > L;
                }
                // smallest (key, list index): a lane visits its indices in
                // ascending order, so a strict comparison keeps its lowest;
                // across lanes three 32-bit reductions give the exact pair
                uint64_t bk = ~0ull;
                uint32_t bkk = 0xFFFFFFFFu;
                for (uint32_t k = lane; k < nl; k += 32) {
                    const uint32_t h = hr[k];
                    const uint64_t w = W[live[k]];
                    uint64_t key;
                    if (rule == DM_RULE_LEAST_LOADED) key = w;
                    else if (affine) key = h == hmax ? w : ~0ull;
                    else key = w + cost * (L - h);
                    if (key < bk || bkk == 0xFFFFFFFFu) { bk = key; bkk = k; }
                }
                const uint32_t khi = __reduce_min_sync(0xffffffffu, (uint32_t)(bk >> 32));
                const uint32_t klo =
                    __reduce_min_sync(0xffffffffu, (uint32_t)(bk >> 32) == khi ? (uint32_t)bk : 0xFFFFFFFFu);
                const uint32_t kk = __reduce_min_sync(
                    0xffffffffu, bk == ((uint64_t(khi) << 32) | klo) ? bkk : 0xFFFFFFFFu);
                if (lane == 0 && kk >= nl) {   // no live instance (the host requires two)
                    set_err(d.err, DM_ERR_NO_INSTANCES);
                    s_ch[rr] = 0xFFFFFFFFu;
                } else if (lane == 0) {
                    const uint32_t ch = live[kk], h = hr[kk];
                    s_t1[rr] = W[s_c1[rr]] + cost * (L - s_h1[rr]);
                    s_t2[rr] = W[s_c2[rr]] + cost * (L - s_h2[rr]);
                    const uint64_t Pold = PT[ch];
                    const uint64_t wa = W[ch] + cost * (L - h);
                    W[ch] = wa;
                    PT[ch] = Pold + (uint64_t(s_nb[rr]) << 32) + 1;
                    s_ch[rr] = ch;
                    s_hch[rr] = h;
                    s_pold[rr] = Pold;
                    s_wa[rr] = wa;
                }
                __syncwarp();
            }
        }
        __syncthreads();
        for (uint32_t rr = threadIdx.x; rr < m; rr += blockDim.x) {
            const uint32_t r = r0 + rr, ch = s_ch[rr], L = s_L[rr], h = s_hch[rr];
            if (ch == 0xFFFFFFFFu) continue;
            const uint64_t Pold = s_pold[rr];
            o.ttft1[r] = s_t1[rr];
            o.ttft2[r] = s_t2[rr];
            o.chosen[r] = ch;
            o.switched[r] = 0;
            d.r_final[r] = ch;
            d.r_touchoff[r] = Pold >> 32;
            ms.tokens += L;
            ms.hits += h;
            ms.est += s_wa[rr] <= slo;
            if (s_t1[rr] > slo && s_t2[rr] > slo) d.info->both_over = 1;
            const uint32_t slot = (uint32_t)Pold;
            if (slot - d.q_head[ch] >= d.Q) {
                set_err(d.err, DM_ERR_CAPACITY);
                continue;
            }
            QEntry e;
            e.seq = seq0 + r;
            e.work = e.remaining = cost * (L - h);
            e.L = L;
            e.c1 = s_c1[rr];
            e.c2 = s_c2[rr];
            e.h1 = s_h1[rr];
            e.h2 = s_h2[rr];
            e.moved = 0;
            e.arrival = t_batch;
            e.koff = 0;
            DM_CHECK(ch < d.M, d.err);
            d.q[uint64_t(ch) * d.Q + (slot & (d.Q - 1))] = e;
        }
    }
    if (cap == 0 && threadIdx.x == 0) set_err(d.err, DM_ERR_CAPACITY);   // not even one request fits
    __syncthreads();
    unsigned __int128 S1 = 0, S2 = 0;
    uint32_t cnt = 0;
    for (uint32_t i = threadIdx.x; i < d.M; i += blockDim.x) {
        d.W[i] = W[i];
        d.q_tail[i] = (uint32_t)PT[i];
        d.log_adv[i] = PT[i] >> 32;
        if (d.inst_state[i] == 1) {
            S1 += W[i];
            S2 += (unsigned __int128)W[i] * W[i];
            ++cnt;
        }
    }
    if (threadIdx.x == 0) d.info->final_dirty = 0;
    finish_metrics(d, n, ms, S1, S2, cnt);
}

cudaError_t launch_choice(const DevState &d, const dm_route_out &o, uint32_t n, uint64_t seq0, uint64_t t_batch,
                          cudaStream_t st) {
    if (n == 0) return cudaSuccess;
    if (d.rule >= DM_RULE_LEAST_LOADED) {
        DM_TRY(launch_carries(d, o, n, st));
        const uint64_t warps = uint64_t(n) * ((d.M + 31) / 32);
        const unsigned grid = (unsigned)std::min<uint64_t>((warps + kAllBlock / 32 - 1) / (kAllBlock / 32), 1u << 30);
        if (uint64_t(n) * d.M <= kPairWarps)
            DM_TRY(launch_pdl(k_probe_pairs, (n * d.M + kAllBlock / 32 - 1) / (kAllBlock / 32), kAllBlock, 0, st, d, n));
        else
            DM_TRY(launch_pdl(k_probe_all, grid, kAllBlock, 0, st, d, n));
        if (d.M <= 64) DM_TRY(launch_choice_all<2>(d, o, n, seq0, t_batch, st));
        else if (d.M <= 128) DM_TRY(launch_choice_all<4>(d, o, n, seq0, t_batch, st));
        else if (d.M <= 256) DM_TRY(launch_choice_all<8>(d, o, n, seq0, t_batch, st));
        else if (d.M <= 512) DM_TRY(launch_choice_all<16>(d, o, n, seq0, t_batch, st));
        else {
            // as much shared memory as the device allows, up to what 1024 requests need
            static SmemOptIn opt;
            static std::atomic<uint32_t> rooms[kDevices];
            int dev = 0;
            DM_TRY(cudaGetDevice(&dev));
            if (dev < 0 || dev >= kDevices) return cudaErrorInvalidDevice;
            uint32_t room = rooms[dev].load(std::memory_order_relaxed);
            if (!room) {
                int optin = 0;
                cudaFuncAttributes fa{};
                DM_TRY(cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
                DM_TRY(cudaFuncGetAttributes(&fa, k_choice_global));
                room = (uint32_t)(size_t(optin) - fa.sharedSizeBytes);
                rooms[dev].store(room, std::memory_order_relaxed);
            }
            const size_t want = global_stage_off(d.M) + size_t(kGlobalReqMax) * (kGlobalReqBytes + 4ull * d.M);
            const uint32_t smem_g = (uint32_t)std::min<size_t>(want, room);
            DM_TRY(opt_in_smem(opt, smem_g, k_choice_global));
            DM_TRY(launch_pdl(k_choice_global, 1, 1024, smem_g, st, d, o, n, seq0, t_batch, smem_g));
        }
        return cudaGetLastError();
    }
    const size_t smem = choice_smem(d.M);
    static SmemOptIn opt;
    DM_TRY(opt_in_smem(opt, smem, k_choice<false>, k_choice<true>));
    // CTA 0 decides; CTAs 1.. sum the batch's segment carries meanwhile (a warp per request)
    constexpr unsigned threads = Pipe<kChoiceChunk>::kThreads, per = threads / 32;
    static const unsigned most = 2 * (unsigned)sm_count();
    const unsigned grid = 1 + std::min((n + per - 1) / per, most);
    if (d.rule == DM_RULE_DUALMAP)
        DM_TRY(launch_pdl(k_choice<false>, grid, threads, smem, st, d, o, n, seq0, t_batch));
    else
        DM_TRY(launch_pdl(k_choice<true>, grid, threads, smem, st, d, o, n, seq0, t_batch));
    return cudaGetLastError();
}


// A batch's outputs into pinned host buffers, one kernel instead of eight copies
// (16 prompts routed from host memory and committed, GB300: 82 and 69 us).
__global__ void k_copy_out(dm_route_out o, dm_route_out w, uint32_t n) {
    pdl_enter();
    const uint32_t r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= n) return;
    w.cand1[r] = o.cand1[r];
    w.cand2[r] = o.cand2[r];
    w.hit1[r] = o.hit1[r];
    w.hit2[r] = o.hit2[r];
    w.ttft1[r] = o.ttft1[r];
    w.ttft2[r] = o.ttft2[r];
    w.chosen[r] = o.chosen[r];
    w.switched[r] = o.switched[r];
}

cudaError_t launch_copy_out(const dm_route_out &o, const dm_route_out &w, uint32_t n, cudaStream_t st) {
    DM_TRY(launch_pdl(k_copy_out, (n + 127) / 128, 128, 0, st, o, w, n));
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Routing with d candidates instead of two (App. A.8,
// "Optimal Candidate Set Size": the paper weighs d and keeps d = 2; this is
// the d-way version of the path, for that comparison).  After the plain
// hashing kernel (f1 chained prefix values and totals):
//   k_route_d   warp per request: segment carries, the d ring positions
//               (function 1 from the prefix values; functions 2..d hash the
//               first K blocks here), a successor search on each ring, the
//               distinct fix, and the leading run of resident blocks on
//               each candidate (4,096 agent prompts, d = 4: 72 us when it
//               walked 32 blocks a round, 50 us by segments);
//   k_choice_d  one CTA: DualMap's SLO-aware rule over d candidates in
//               arrival order (the choice pipeline), queue appends, the
//               commit's per-request offsets and the batch's metrics,
//               exactly as k_choice leaves them for d = 2.


// Index (level 0) of the successor of p on ring f.  Whole warp.
__device__ __forceinline__ uint32_t ring_search1(const DevState &d, int f, uint64_t p, int lane) {
    const int top = (int)d.nlev - 1;
    const uint64_t nt = d.lev_n[top];
    const uint64_t vt = (uint64_t)lane < nt ? level_ptr(d, f, top)[lane] : ~0ull;
    int64_t i = (int64_t)__popc(__ballot_sync(0xffffffffu, vt < p)) - 1;
    for (int k = top - 1; k >= 0; --k) {
        const uint64_t nk = d.lev_n[k];
        const uint64_t a = (uint64_t)(i < 0 ? 0 : i) * 32 + lane;
        const uint64_t v = (i >= 0 && a < nk) ? level_ptr(d, f, k)[a] : ~0ull;
        const int c = __popc(__ballot_sync(0xffffffffu, v < p));
        if (i >= 0) i = i * 32 + c - 1;
    }
    return (uint32_t)(i + 1 == (int64_t)d.R ? 0 : i + 1);
}

// NH key word j of function f (0-based).
__device__ __forceinline__ uint32_t nh_key(const DevState &d, uint32_t f, uint32_t j) {
    return f == 0 ? d.K1[j] : f == 1 ? d.K2[j] : d.Kx[(f - 2) * 64 + j];
}

__global__ void k_route_d(DevState d, const uint32_t *tokens, uint32_t n) {
    pdl_enter();
    if (has_err(d.err)) return;
    const int lane = threadIdx.x & 31;
    const uint32_t r = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (r >= n) return;
    request_carries(d, r, lane);
    __syncwarp();
    const uint32_t nblk = d.r_nblk[r], s0 = d.r_segoff[r], B = d.B, nd = d.nd;
    const uint64_t bo = d.r_blkoff[r];
    const uint32_t K = min(d.Kroute, nblk);
    const uint32_t *tok = tokens + d.r_tokoff[r];
    uint32_t cand[kMaxD];
    for (uint32_t f = 0; f < nd; ++f) {
        uint64_t P;
        if (f == 0) {
            P = d.plocal[bo + K - 1] + d.seg_carry[s0 + (K - 1) / kSegBlocks];
        } else {   // function f over the first K blocks: a lane per block
            const uint64_t G = f == 1 ? d.G2 : d.Gx[f - 2];
            uint64_t acc = 0;
            for (uint32_t b = lane; b < K; b += 32) {
                uint64_t nh = 0;
                for (uint32_t i = 0; i < B; i += 2)
                    nh += uint64_t(tok[uint64_t(b) * B + i] + nh_key(d, f, i)) *
                          uint64_t(tok[uint64_t(b) * B + i + 1] + nh_key(d, f, i + 1));
                acc += fmix64(nh + uint64_t(b + 1) * G);
            }
            P = warp_sum_u64(acc);
        }
        const uint64_t Sr = f == 0 ? d.Sr1 : f == 1 ? d.Sr2 : d.Srx[f - 2];
        uint32_t x = d.ring[f].owner[ring_search1(d, (int)f, fmix64(P ^ Sr), lane)];
        for (uint32_t k = 0; k < nd; ++k) {   // taken by an earlier ring: the next live id after it
            bool taken = false;
            for (uint32_t g = 0; g < f; ++g) taken |= cand[g] == x;
            if (!taken) break;
            x = d.next_live[x];
        }
        cand[f] = x;
    }
    // leading run of resident blocks on each candidate (index as of the start
    // of the batch), two candidates at a time: the first block of every
    // segment, 32 segments a round, then the segment that holds the run's end
    const uint64_t mask = d.S - 1;
    const uint32_t nseg = (nblk + kSegBlocks - 1) / kSegBlocks;
    for (uint32_t f0 = 0; f0 < nd; f0 += 2) {
        const bool two = f0 + 1 < nd;
        const uint32_t ca = cand[f0], cb = two ? cand[f0 + 1] : ca;
        const Slot *const t[2] = {d.table[ca], d.table[cb]};
        const uint64_t front[2] = {d.log_front[ca], d.log_front[cb]};
        uint32_t js[2] = {nseg, two ? nseg : 0}, m[2];   // first segment whose first block is missing
        bool open[2] = {true, two};
        for (uint32_t g0 = 0; g0 < nseg && (open[0] || open[1]); g0 += 32) {
            const uint32_t sg = g0 + lane;
            const uint64_t key[1] = {
                sg < nseg ? cache_key(d.plocal[bo + uint64_t(sg) * kSegBlocks] + d.seg_carry[s0 + sg], d.Sc) : 0};
            const uint64_t home[1] = {group_home(key[0], 0, mask)};   // a segment's first block anchors its own group
            Slot s[2];
            int look[2][1];
#pragma unroll
            for (int x = 0; x < 2; ++x) s[x] = sg < nseg && open[x] ? load_slot(t[x] + home[0]) : Slot{0, 0};
#pragma unroll
            for (int x = 0; x < 2; ++x) look[x][0] = sg < nseg ? look_at(s[x], key[0], front[x]) : kOut;
            uint32_t run[2];
            leading_runs<2, 1>(look, t, front, mask, key, home, lane, d.err, d.loop_limit, run);
#pragma unroll
            for (int x = 0; x < 2; ++x)
                if (open[x] && run[x] < min(32u, nseg - g0)) {
                    js[x] = g0 + run[x];
                    open[x] = false;
                }
        }
#pragma unroll
        for (int x = 0; x < 2; ++x) m[x] = min(js[x] * kSegBlocks, nblk);
#pragma unroll 1
        for (int x = 0; x < 2; ++x) {
            if (js[x] == 0 || (x == 1 && js[1] == js[0])) continue;
            const uint32_t c0 = (js[x] - 1) * kSegBlocks, cn = min(kSegBlocks, nblk - c0);
            const uint64_t carry = d.seg_carry[s0 + js[x] - 1];
            uint64_t key[2], home[2];
            Slot s[2][2];
            int look[2][2];
            const bool in[2] = {x == 0, js[1] == js[x]};
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                const uint32_t e = 32 * q + lane;
                key[q] = e < cn ? cache_key(d.plocal[bo + c0 + e] + carry, d.Sc) : 0;
                home[q] = group_home(group_anchor(key[q], lane), c0 + e, mask);
#pragma unroll
                for (int y = 0; y < 2; ++y) s[y][q] = e < cn && in[y] ? load_slot(t[y] + home[q]) : Slot{0, 0};
            }
#pragma unroll
            for (int q = 0; q < 2; ++q)
#pragma unroll
                for (int y = 0; y < 2; ++y) look[y][q] = 32u * q + lane < cn ? look_at(s[y][q], key[q], front[y]) : kOut;
            uint32_t run[2];
            leading_runs<2, 2>(look, t, front, mask, key, home, lane, d.err, d.loop_limit, run);
#pragma unroll
            for (int y = 0; y < 2; ++y)
                if (in[y] && run[y] < cn) m[y] = c0 + run[y];
        }
        if (lane == 0) {
            d.rd_cand[uint64_t(r) * nd + f0] = ca;
            d.rd_hit[uint64_t(r) * nd + f0] = m[0] * B;
            if (two) {
                d.rd_cand[uint64_t(r) * nd + f0 + 1] = cb;
                d.rd_hit[uint64_t(r) * nd + f0 + 1] = m[1] * B;
            }
        }
    }
    if (lane == 0) d.r_K[r] = K;
}

// Staging of one chunk: candidates, uncached work on each, the load of each
// as the request found it, which candidates have the most hit tokens.
template <uint32_t ND, uint32_t kChunk>
struct ChoiceStageD {
    uint64_t u[ND][kChunk], Wf[ND][kChunk];
    uint16_t c[ND][kChunk];
    uint8_t most[kChunk];             // bit f: candidate f has the most hit tokens
    uint8_t lev[kChunk], pick[kChunk], over[kChunk];
    uint32_t wsum[kChunk / 32];       // per window: sum of the largest works, in units of 2^kWorkShift (rounded up)
    uint32_t u32[ND][kChunk];         // low words of u
    uint16_t from[ND][kChunk];        // word of the exchange rows that holds candidate f's load
    uint8_t last[kChunk];             // bit f: no later request of the window names candidate f
    uint32_t nlev[kChunk / 32];
};
constexpr uint64_t kSmallD = 1ull << 28;   // loads below it are decided in 32 bits, a candidate's number beside them
// Exchange rows: for each lane what its request leaves on its candidates, then
// the loads it found at the window's start; twice, written and read in turn.
constexpr uint32_t exchange_stride(uint32_t nd) { return nd > 4 ? 8 : nd > 2 ? 4 : nd; }
constexpr uint32_t exchange_words(uint32_t nd) { return 2 * 32 * exchange_stride(nd); }   // of one of the two
constexpr uint32_t choice_d_chunk(uint32_t nd) { return nd <= 4 ? 256 : 128; }   // three buffers beside 8,192 instances

// DualMap's rule over ND candidates, in arrival order (the pipeline above),
// then the batch's loads, queue tails, commit offsets and metrics as
// k_choice leaves them.  Dynamic shared memory: W and the packed (records
// << 32 | queue tail) counter of every instance, then the staging buffers.
template <uint32_t ND>
__global__ void __launch_bounds__(Pipe<choice_d_chunk(ND)>::kThreads, 1) k_choice_d(DevState d, dm_route_out_d o,
                                                                                 uint32_t n, uint64_t seq0,
                                                                                 uint64_t t_batch) {
    pdl_enter();
    extern __shared__ __align__(16) unsigned char smem[];
    if (has_err(d.err)) return;
    constexpr uint32_t kChunk = choice_d_chunk(ND);
    using Stage = ChoiceStageD<ND, kChunk>;
    uint64_t *W = reinterpret_cast<uint64_t *>(smem);
    uint64_t *PT = W + d.M;
    Stage *const SB = reinterpret_cast<Stage *>(PT + d.M);
    constexpr uint32_t kStride = exchange_stride(ND);
    __shared__ alignas(16) uint32_t X[2 * exchange_words(ND)];
    const int lane = threadIdx.x & 31;
    uint32_t live_bits = 0;   // bit k: instance threadIdx.x + k * blockDim.x is live (M <= 32 * 352)
    for (uint32_t i = threadIdx.x, k = 0; i < d.M; i += blockDim.x, ++k) {
        W[i] = d.W[i];
        PT[i] = d.q_tail[i];
        live_bits |= uint32_t(d.inst_state[i] == 1) << k;
    }
    const uint64_t cost = d.cost, slo = d.slo;
    MetricSums ms{0, 0, 0, 0};

    auto stage = [&](uint32_t buf, uint32_t k, uint32_t m, uint32_t base) {
        if ((k & ~31u) >= m) return;   // no request in this window
        Stage &S = SB[buf];
        const bool valid = k < m;
        uint32_t ids[ND];
#pragma unroll
        for (uint32_t f = 0; f < ND; ++f) ids[f] = kNone;
        uint64_t umax = 0;
        if (valid) {
            const uint32_t r = base + k, L = d.r_L[r];
            const uint32_t *c = d.rd_cand + uint64_t(r) * ND, *h = d.rd_hit + uint64_t(r) * ND;
            uint32_t cf[ND], hf[ND], hmax = 0;
#pragma unroll
            for (uint32_t f = 0; f < ND; ++f) {
                cf[f] = c[f];
                hf[f] = h[f];
                hmax = max(hmax, hf[f]);
            }
            uint32_t most = 0;
#pragma unroll
            for (uint32_t f = 0; f < ND; ++f) {
                S.u[f][k] = cost * (L - hf[f]);
                S.u32[f][k] = (uint32_t)S.u[f][k];
                umax = max(umax, cost * (L - hf[f]));
                most |= uint32_t(hf[f] == hmax) << f;
                ids[f] = cf[f];
                o.cand[uint64_t(r) * ND + f] = cf[f];
                o.hit[uint64_t(r) * ND + f] = hf[f];
            }
            S.most[k] = (uint8_t)most;
        }
        uint32_t lev, nlev, from[ND];
        S.last[k] = (uint8_t)window_links<ND, kStride>(ids, valid, lane, from, lev, nlev);
        S.lev[k] = valid ? (uint8_t)lev : kNoLevel;
#pragma unroll
        for (uint32_t f = 0; f < ND; ++f) {
            S.c[f][k] = valid ? (uint16_t)ids[f] : 0;   // every lane of a window reads its loads
            S.from[f][k] = (uint16_t)(valid && from[f] != kNone ? from[f] : (32 + lane) * kStride + f);
        }
        const uint32_t sum = __reduce_add_sync(0xffffffffu, (uint32_t)((min(umax, kSmallD) + kWorkUnit) >> kWorkShift));
        if (lane == 0) {
            S.nlev[k / 32] = nlev;
            S.wsum[k / 32] = sum;
        }
    };

    // one chunk whose loads stay below 2^28, as in k_choice: every lane decides
    // its request at every level.  The loads pass between the lanes through
    // shared memory (a row per lane).  A candidate's key is its load and its
    // number, so one minimum over the candidates gives the least loaded and
    // the earlier ring on ties; the candidates with the most hit tokens have
    // the same uncached work.
    uint64_t bound = 0;   // no load exceeds it, unless it is kSmallD
    struct Win {
        uint32_t nlev, most, last, c[ND], u[ND], from[ND];
    };
    auto window = [&](const Stage &S, uint32_t w0) {
        const uint32_t k = w0 + lane;
        Win x;
        x.nlev = S.nlev[w0 / 32];
        x.most = S.most[k];
        x.last = S.last[k];
#pragma unroll
        for (uint32_t f = 0; f < ND; ++f) {
            x.c[f] = S.c[f][k];
            x.u[f] = S.u32[f][k];   // past the batch's end: unused
            x.from[f] = S.from[f][k];
        }
        return x;
    };
    auto begin = [&] {
        for (uint32_t i = lane; i < d.M; i += 32) bound = max(bound, min(d.W[i], kSmallD));
        bound = __reduce_max_sync(0xffffffffu, (uint32_t)bound);
    };
    auto decide32 = [&](Stage &S, uint32_t m) {
        volatile uint32_t *const W32 = reinterpret_cast<volatile uint32_t *>(W);   // low words; the high ones are 0
        constexpr uint32_t kRow = exchange_words(ND);
        Win nx = window(S, 0);
        for (uint32_t w0 = 0; w0 < m; w0 += 32) {
            const Win x = nx;
            uint32_t w[ND];
#pragma unroll
            for (uint32_t f = 0; f < ND; ++f) {
                w[f] = W32[2 * x.c[f]];
                X[(32 + lane) * kStride + f] = w[f];
                X[kRow + (32 + lane) * kStride + f] = w[f];
            }
            nx = window(S, w0 + 32 < m ? w0 + 32 : 0);
            // a misses the SLO iff its key > late (never when all hits are equal)
            uint32_t ua = 0, skip[ND];
#pragma unroll
            for (uint32_t f = 0; f < ND; ++f) {
                const bool in = (x.most >> f) & 1u;
                ua = in ? x.u[f] : ua;
                skip[f] = in ? 0u : 0x7FFFFFFFu;
            }
            const int32_t late = x.most == (1u << ND) - 1u ? INT32_MAX
                                 : ua > slo               ? -1
                                                          : (int32_t)(min(slo - ua, kSmallD - 1) * 8 + 7);
            uint32_t key, out[ND], row = 0;
            int32_t over;   // all ones: a misses the SLO and some candidate has fewer hits
            auto step = [&] {
                uint32_t kf[ND], ka[ND], km[ND];
#pragma unroll
                for (uint32_t f = 0; f < ND; ++f) {
                    kf[f] = km[f] = w[f] * 8 + f;
                    ka[f] = kf[f] | skip[f];
                }
#pragma unroll
                for (uint32_t s = 1; s < ND; s *= 2)
#pragma unroll
                    for (uint32_t f = 0; f + s < ND; f += 2 * s) {
                        ka[f] = min(ka[f], ka[f + s]);
                        km[f] = min(km[f], km[f + s]);
                    }
                over = (late - (int32_t)ka[0]) >> 31;
                const int32_t move = over & ((int32_t)(km[0] - (ka[0] & ~7u)) >> 31);   // the least loaded is below a
                key = ka[0] ^ ((ka[0] ^ km[0]) & (uint32_t)move);
#pragma unroll
                for (uint32_t f = 0; f < ND; ++f) out[f] = w[f] + (key == kf[f] ? x.u[f] : 0u);
            };
            const uint32_t nlev = __reduce_max_sync(0xffffffffu, x.nlev);   // uniform: the loop below has no divergence
            step();
            for (uint32_t l = 1; l < nlev; ++l) {
#pragma unroll
                for (uint32_t f = 0; f < ND; ++f) X[row + lane * kStride + f] = out[f];
                __syncwarp();
#pragma unroll
                for (uint32_t f = 0; f < ND; ++f) w[f] = X[row + x.from[f]];
                row ^= kRow;
                step();
            }
#pragma unroll
            for (uint32_t f = 0; f < ND; ++f)
                if ((x.last >> f) & 1u) W32[2 * x.c[f]] = out[f];
            __syncwarp();
            const uint32_t k = w0 + lane;
#pragma unroll
            for (uint32_t f = 0; f < ND; ++f) S.Wf[f][k] = w[f];
            S.pick[k] = (uint8_t)(key & 7u);
            S.over[k] = over != 0;
        }
    };

    auto decide = [&](uint32_t buf, uint32_t m) {
        Stage &S = SB[buf];
        bound = min(bound + (uint64_t(__reduce_add_sync(0xffffffffu, (uint32_t)lane < (m + 31) / 32 ? S.wsum[lane] : 0))
                             << kWorkShift),
                    kSmallD);
        if (bound < kSmallD) {
            decide32(S, m);
            return;
        }
        volatile uint64_t *const Wv = W;
        for (uint32_t w0 = 0; w0 < m; w0 += 32) {
            const uint32_t k = w0 + lane;
            const uint32_t mine = S.lev[k], nlev = S.nlev[w0 / 32], most = S.most[k];
            uint32_t c[ND];
            uint64_t u[ND], oW[ND];
            uint32_t opick = 0;
            bool oover = false;
#pragma unroll
            for (uint32_t f = 0; f < ND; ++f) {
                c[f] = mine != kNoLevel ? S.c[f][k] : 0;
                u[f] = S.u[f][k];   // past the batch's end: unused
                oW[f] = 0;
            }
            for (uint32_t l = 0; l < nlev; ++l) {
                uint64_t w[ND];
#pragma unroll
                for (uint32_t f = 0; f < ND; ++f) w[f] = Wv[c[f]];
                // a: the least loaded of those with the most hit tokens (tie: the earlier ring)
                uint64_t wa = ~0ull, ua = 0, wm = ~0ull, um = 0;
                uint32_t a = ND, cm = 0, fm = 0, ca = 0;
#pragma unroll
                for (uint32_t f = 0; f < ND; ++f) {
                    const bool ta = ((most >> f) & 1u) && (a == ND || w[f] < wa);
                    wa = ta ? w[f] : wa;
                    ua = ta ? u[f] : ua;
                    ca = ta ? c[f] : ca;
                    a = ta ? f : a;
                    const bool tm = f == 0 || w[f] < wm;
                    wm = tm ? w[f] : wm;
                    um = tm ? u[f] : um;
                    cm = tm ? c[f] : cm;
                    fm = tm ? f : fm;
                }
                // over: some candidate has fewer hits and a misses the SLO; then
                // the least loaded of all (tie: a, then the earlier ring)
                const bool over = most != (1u << ND) - 1u && wa + ua > slo;
                const bool mv = over && wm < wa;
                if (mine == l) {
                    Wv[mv ? cm : ca] = mv ? wm + um : wa + ua;
#pragma unroll
                    for (uint32_t f = 0; f < ND; ++f) oW[f] = w[f];
                    opick = mv ? fm : a;
                    oover = over;
                }
                __syncwarp();
            }
#pragma unroll
            for (uint32_t f = 0; f < ND; ++f) S.Wf[f][k] = oW[f];
            S.pick[k] = (uint8_t)opick;
            S.over[k] = oover;
        }
    };

    auto emit = [&](uint32_t buf, uint32_t k, uint32_t m, uint32_t base) {
        const Stage &S = SB[buf];
        const bool valid = k < m;
        const uint32_t r = base + k, pick = valid ? S.pick[k] : 0;
        const uint32_t ch = valid ? S.c[pick][k] : 0;
        const uint32_t nbr = valid ? d.r_nblk[r] : 0, L = valid ? d.r_L[r] : 0, qh = d.q_head[ch];
        const uint64_t pt = record_place<kChunk>(PT, ch, (uint64_t(nbr) << 32) + 1, valid, k / 32, (m + 31) / 32,
                                                 lane);
        if (!valid) return;
        bool all_over = true;
#pragma unroll
        for (uint32_t f = 0; f < ND; ++f) {
            const uint64_t t = S.Wf[f][k] + S.u[f][k];
            o.ttft[uint64_t(r) * ND + f] = t;
            all_over = all_over && t > slo;
        }
        if (all_over) d.info->both_over = 1;
        o.chosen[r] = ch;
        o.switched[r] = S.over[k];
        d.r_final[r] = ch;
        d.r_touchoff[r] = pt >> 32;   // offset among this batch's records of ch
        const uint32_t *h = d.rd_hit + uint64_t(r) * ND;
        ms.tokens += L;
        ms.hits += h[pick];
        ms.sw += S.over[k];
        ms.est += S.Wf[pick][k] + S.u[pick][k] <= slo;
        const uint32_t slot = (uint32_t)pt;
        if (slot - qh >= d.Q) {
            set_err(d.err, DM_ERR_CAPACITY);
            return;
        }
        QEntry e;
        e.seq = seq0 + r;
        e.work = e.remaining = S.u[pick][k];
        e.L = L;
        e.c1 = S.c[0][k];
        e.c2 = S.c[ND > 1 ? 1 : 0][k];
        e.h1 = h[0];
        e.h2 = h[ND > 1 ? 1 : 0];
        e.moved = 0;
        e.arrival = t_batch;
        e.koff = 0;
        DM_CHECK(ch < d.M, d.err);
        d.q[uint64_t(ch) * d.Q + (slot & (d.Q - 1))] = e;
    };

    // (W and PT are first read after the first chunk's barrier)
    choice_pipeline<kChunk, kChunk>(n, begin, stage, decide, emit);
    unsigned __int128 S1 = 0, S2 = 0;
    uint32_t cnt = 0;
    for (uint32_t i = threadIdx.x, k = 0; i < d.M; i += blockDim.x, ++k) {
        d.W[i] = W[i];
        d.q_tail[i] = (uint32_t)PT[i];
        d.log_adv[i] = PT[i] >> 32;
        if ((live_bits >> k) & 1u) {
            S1 += W[i];
            S2 += (unsigned __int128)W[i] * W[i];
            ++cnt;
        }
    }
    if (threadIdx.x == 0) d.info->final_dirty = 0;
    finish_metrics(d, n, ms, S1, S2, cnt);
}

template <uint32_t ND>
static cudaError_t launch_choice_d(const DevState &d, const dm_route_out_d &o, uint32_t n, uint64_t seq0,
                                   uint64_t t_batch, cudaStream_t st) {
    constexpr uint32_t kChunk = choice_d_chunk(ND);
    const size_t smem = size_t(d.M) * 16 + 3 * sizeof(ChoiceStageD<ND, kChunk>);
    static SmemOptIn opt;
    DM_TRY(opt_in_smem(opt, smem, k_choice_d<ND>));
    return launch_pdl(k_choice_d<ND>, 1, Pipe<kChunk>::kThreads, smem, st, d, o, n, seq0, t_batch);
}

cudaError_t launch_route_d(const DevState &d, const dm_batch &b, const dm_route_out_d &o, uint64_t seq0,
                           cudaStream_t st) {
    if (b.n == 0) return cudaSuccess;
    DM_TRY(launch_pdl(k_route_d, (b.n + 7) / 8, 256, 0, st, d, b.tokens, b.n));
    switch (d.nd) {
        case 1: DM_TRY(launch_choice_d<1>(d, o, b.n, seq0, b.batch_time_us, st)); break;
        case 2: DM_TRY(launch_choice_d<2>(d, o, b.n, seq0, b.batch_time_us, st)); break;
        case 3: DM_TRY(launch_choice_d<3>(d, o, b.n, seq0, b.batch_time_us, st)); break;
        case 4: DM_TRY(launch_choice_d<4>(d, o, b.n, seq0, b.batch_time_us, st)); break;
        case 5: DM_TRY(launch_choice_d<5>(d, o, b.n, seq0, b.batch_time_us, st)); break;
        case 6: DM_TRY(launch_choice_d<6>(d, o, b.n, seq0, b.batch_time_us, st)); break;
        case 7: DM_TRY(launch_choice_d<7>(d, o, b.n, seq0, b.batch_time_us, st)); break;
        case 8: DM_TRY(launch_choice_d<8>(d, o, b.n, seq0, b.batch_time_us, st)); break;
        default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

}  // namespace dm
