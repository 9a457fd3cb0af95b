// osd_verify.cu -- speculative-sampling verification (Section 3 and
// Appendix A.1 of the paper; the verify step of Algorithm 1) on sm_103a.
//
// T > 0: one launch, a thread-block cluster per sequence, each CTA owning a span of
// the vocabulary.  The tests u_i < p_i(y_i)/q_i(y_i) run in order and the first failure
// ends them, so the rows past it decide nothing:
//
//   verify_lazy_kernel   rounds of positions: the round's rows are streamed once, the
//                        span statistics (max and sum of exp((x - max)/T)) meet over the
//                        cluster by st.async, every CTA runs the round's tests, and
//                        only a round without a failure asks for the next one's rows.
//   verify_fused_kernel  small batches, where latency costs more than bytes: all 2k + 1
//                        rows staged in shared memory, one round.
//
// The extra token is then drawn from norm(max(0, p_a - q_a)) (or p_k when all k
// pass) by inverse CDF: each CTA sums the residual weights of its span per
// sub-tile, the span totals meet as exact 64-bit fixed point, and the CTA whose
// span holds u*W rescans that one sub-tile exactly.
//
// T = 0: two launches, row_argmax_kernel (the argmax of every target row's slices) and
// verify_greedy_kernel, one warp per sequence: the matches in order, the target
// argmax at the first mismatch; large batches walk on demand (greedy_walk_kernel).
//
// The log-ratio of the accept test is formed from differences of raw logits and
// maxima, (t_y - m_t) - (z_y - m_z), and the ratio of the two sums, so no
// log-sum-exp is rounded on its own.
#include <cuda.h>

#include <algorithm>
#include <climits>
#include <cstdint>
#include <mutex>
#include <type_traits>

#include "osd.h"
#include "osd_device.cuh"
#include "osd_host.hpp"
#include "osd_rowstats.cuh"

namespace osd {

constexpr int kFinUnroll = 4;     // sub-tiles of loads in flight per warp
// Where the draw reads the rows from: shared memory, 16-byte-aligned rows in global
// memory, or rows of any alignment there.
constexpr int kRowsStaged = 0, kRowsAligned = 1, kRowsAny = 2;

struct FinParams {
    const void* draft;
    const void* target;
    int B, k, V;
    const int32_t* tokens;
    const float* uniforms;
    float T, c_hi, c_lo;
    const RowStat* stats;
    int n_slices;
    int32_t* accepted;
    int32_t* out_tokens;
    uint8_t* mask;
    float* diag_margin;
    float* diag_gap;
    int csize;  // CTAs per sequence (cluster size)
    int span;   // vocabulary entries per CTA of the cluster
};


// T = 0: the accept tests are argmax matches, and the extra token is the target
// argmax at the first mismatch.  One warp per sequence, a small kernel of its
// own: at serving batch sizes this pass is latency-bound, and a compact kernel
// starts faster than the sampling kernel with its greedy branch would.
constexpr int kGreedyWarps = 4;
__global__ void __launch_bounds__(kGreedyWarps * 32) verify_greedy_kernel(FinParams p) {
    const int lane = threadIdx.x & 31;
    const int b = blockIdx.x * kGreedyWarps + (threadIdx.x >> 5);
    if (b >= p.B) return;
    const int k = p.k, V = p.V;
    const int32_t* y = p.tokens + size_t(b) * k;
    // the draft tokens before the statistics are needed (one round of loads)
    constexpr int kC = (OSD_VERIFY_MAX_K + 1 + 31) / 32;
    int yv[kC];
    bool bad = false;
#pragma unroll
    for (int c = 0; c < kC; ++c) {
        const int i = c * 32 + lane;
        yv[c] = (i < k) ? y[i] : 0;
        bad |= (i < k) && (yv[c] < 0 || yv[c] >= V);
    }
    grid_dependency_sync();  // the row statistics are complete from here on
    // row i <= k of the sequence: its target argmax, lowest index on ties, merged
    // from the slices by the lane that owns the row
    int idx[kC];
    unsigned fail = 0;
    int a = k;
#pragma unroll
    for (int c = 0; c < kC; ++c) {
        const int i = c * 32 + lane;
        idx[c] = 0;
        if (i <= k) {
            const RowStat* st = p.stats + ((long long)b * (k + 1) + i) * p.n_slices;
            MaxIdx acc{kNegInf, INT_MAX};
            for (int sl = 0; sl < p.n_slices; ++sl) acc = merge_mi(acc, MaxIdx{st[sl].m, st[sl].idx});
            idx[c] = (acc.i == INT_MAX) ? 0 : acc.i;
        }
        fail = __ballot_sync(0xffffffffu, i < k && yv[c] != idx[c]);
        if (fail && a == k) a = c * 32 + __ffs(fail) - 1;
    }
    bad = __any_sync(0xffffffffu, bad);
    int32_t* out = p.out_tokens + size_t(b) * (k + 1);
    if (lane == 0) {
        p.accepted[b] = bad ? -1 : a;
        if (p.diag_gap) p.diag_gap[b] = __int_as_float(0x7fc00000);
    }
    // the token at a is the target argmax there, held by lane a % 32 in slot a / 32
    int at = 0;
#pragma unroll
    for (int c = 0; c < kC; ++c) {
        const int v = __shfl_sync(0xffffffffu, idx[c], a & 31);
        if (c == a / 32) at = v;
    }
#pragma unroll
    for (int c = 0; c < kC; ++c) {
        const int i = c * 32 + lane;
        if (i <= k) out[i] = bad ? -1 : (i < a ? yv[c] : (i == a ? at : -1));
        if (i < k) {
            p.mask[size_t(b) * k + i] = (!bad && i == a) ? 1 : 0;
            if (p.diag_margin) p.diag_margin[size_t(b) * k + i] = __int_as_float(0x7fc00000);
        }
    }
}

// The same walk on demand (osd_rowstats.cuh): position i follows position i - 1 by draft token i - 1.
struct GreedyChain {
    FinParams p;
    __device__ bool node_ok(int b) const {
        bool ok = true;
        for (int i = threadIdx.x; i < p.k; i += kWalkThreads) {
            const int y = p.tokens[size_t(b) * p.k + i];
            ok = ok && y >= 0 && y < p.V;
        }
        return ok;
    }
    __device__ size_t row(int b, int i) const { return size_t(b) * (p.k + 1) + i; }
    __device__ int next(int i) const { return i < p.k ? i + 1 : -1; }
    __device__ int child(int b, int i, int x) const { return i < p.k && p.tokens[size_t(b) * p.k + i] == x ? i + 1 : -1; }
    __device__ void step(int, int, int) const {}
    __device__ void finish(int b, int a, int, int x) const {
        if (threadIdx.x == 0) {
            p.accepted[b] = a;
            if (p.diag_gap) p.diag_gap[b] = __int_as_float(0x7fc00000);
        }
        for (int i = threadIdx.x; i <= p.k; i += kWalkThreads)
            p.out_tokens[size_t(b) * (p.k + 1) + i] = i < a ? p.tokens[size_t(b) * p.k + i] : (i == a ? x : -1);
        for (int i = threadIdx.x; i < p.k; i += kWalkThreads) {
            p.mask[size_t(b) * p.k + i] = i == a ? 1 : 0;
            if (p.diag_margin) p.diag_margin[size_t(b) * p.k + i] = __int_as_float(0x7fc00000);
        }
    }
    __device__ void bad(int b) const;
};

// Shared memory of one sequence's decision: the merged statistics of its 2k+1
// rows (local row r <= k is target row r, r > k is draft row r-k-1), the draft
// tokens, the two logits each accept test needs, the uniforms, and a.
struct SeqSmem {
    float m[2 * OSD_VERIFY_MAX_K + 1];
    float s[2 * OSD_VERIFY_MAX_K + 1];
    float zy[OSD_VERIFY_MAX_K], ty[OSD_VERIFY_MAX_K];
    int y[OSD_VERIFY_MAX_K];
    float u[OSD_VERIFY_MAX_K + 1];
};

// Outputs of a sequence with a bad draft token (one CTA of kThreads writes them).
template <int kThreads>
__device__ __forceinline__ void seq_write_bad(const FinParams& p, int b) {
    const int tid = threadIdx.x, k = p.k;
    int32_t* out = p.out_tokens + size_t(b) * (k + 1);
    if (tid == 0) { p.accepted[b] = -1; if (p.diag_gap) p.diag_gap[b] = __int_as_float(0x7fc00000); }
    for (int i = tid; i <= k; i += kThreads) out[i] = -1;
    for (int i = tid; i < k; i += kThreads) {
        p.mask[size_t(b) * k + i] = 0;
        if (p.diag_margin) p.diag_margin[size_t(b) * k + i] = __int_as_float(0x7fc00000);
    }
}
__device__ void GreedyChain::bad(int b) const { seq_write_bad<kWalkThreads>(p, b); }

// One round of accept tests, run by warp 0 of every CTA of the cluster alike:
// positions i0 .. i0 + w - 1, a lane each, the first failing one is a.  Returns
// a, k when the bonus position is reached without a failure, or -1 when the
// round ends undecided; writes the margins of the decided positions when `margins`.
__device__ __forceinline__ int seq_test(const FinParams& p, int b, const SeqSmem& sh, int i0, int w, bool margins) {
    const int lane = threadIdx.x & 31, k = p.k;
    for (int c = 0; c < w; c += 32) {
        const int i = i0 + c + lane;
        const bool test = c + lane < w && i < k;
        float ratio = 0.f;
        bool fail = false;
        if (test) {
            const float D = (sh.ty[i] - sh.m[i]) - (sh.zy[i] - sh.m[k + 1 + i]);
            ratio = expf(__fdiv_rn(D, p.T)) * __fdiv_rn(sh.s[k + 1 + i], sh.s[i]);
            fail = !(sh.u[i] < ratio);
        }
        const unsigned f = __ballot_sync(0xffffffffu, fail);
        const int a = f ? i0 + c + __ffs(f) - 1 : k;
        if (margins && test && i <= a) p.diag_margin[size_t(b) * k + i] = fabsf(sh.u[i] - ratio);
        if (f) return a;
    }
    return i0 + w == k + 1 ? k : -1;
}

// Warp 0, after a round's span statistics (nr rows, `parts` <= kMostParts partials each): merge
// them, push the span's to every CTA of the cluster (slot [rank][row] of recv,
// completing on bar), merge the cluster's and run the tests.  Every CTA merges the
// same slots in the same order, so all decide alike.  Returns seq_test's answer,
// or -2 when a CTA's copies (`stuck`, sent as a negative sum) or the wait gave up.
template <int kMostParts>
__device__ __forceinline__ int seq_round(const FinParams& p, int b, SeqSmem& sh, const MaxSum* part, int parts,
                                         MaxSum* recv, int stride, uint64_t* bar, uint32_t parity, int rank, int i0,
                                         int w, int nr, bool stuck) {
    const int lane = threadIdx.x & 31, csize = p.csize, k = p.k;
    const float ch = p.c_hi, cl = p.c_lo;
    for (int r = lane; r < nr; r += 32) {
        MaxSum acc = merge_slots<kMostParts>(part + r * parts, 1, parts, ch, cl);
        if (stuck) acc.s = -1.f;
        if (csize > 1) {
            for (int d = 0; d < csize; ++d)
                st_async_v2(map_rank(&recv[rank * stride + r], static_cast<uint32_t>(d)), make_float2(acc.m, acc.s),
                            map_rank(bar, static_cast<uint32_t>(d)));
        } else {
            recv[r] = acc;
        }
    }
    bool gone = false;
    if (csize > 1) {
        if (lane == 0) mbar_arrive_expect_tx(bar, static_cast<uint32_t>(csize * nr) * 8u);
        gone = !mbar_wait_cluster_bounded(bar, parity, kPeerWaitNs);
    }
    __syncwarp();
    if (!gone) {
        for (int r = lane; r < nr; r += 32) {
            for (int c = 0; c < csize; ++c) gone |= recv[c * stride + r].s < 0.f;
            const MaxSum o = merge_slots<kSeqMaxCluster>(recv + r, stride, csize, ch, cl);
            const int at = (r < w) ? i0 + r : k + 1 + i0 + r - w;
            sh.m[at] = o.m;
            sh.s[at] = o.s;
        }
    }
    if (__any_sync(0xffffffffu, gone)) return -2;
    return seq_test(p, b, sh, i0, w, rank == 0 && p.diag_margin);
}

// accepted, the accepted tokens and the -1 padding after a, the mask, and the
// margins past the decision (one CTA of kThreads); the token at a is the draw's.
template <int kThreads>
__device__ __forceinline__ void seq_write_outputs(const FinParams& p, int b, const SeqSmem& sh, int a) {
    const int tid = threadIdx.x, k = p.k;
    int32_t* out = p.out_tokens + size_t(b) * (k + 1);
    if (tid == 0) p.accepted[b] = a;
    for (int i = tid; i <= k; i += kThreads)
        if (i < a) out[i] = sh.y[i];
        else if (i > a) out[i] = -1;
    for (int i = tid; i < k; i += kThreads) {
        p.mask[size_t(b) * k + i] = (i == a) ? 1 : 0;
        if (p.diag_margin && i > a) p.diag_margin[size_t(b) * k + i] = __int_as_float(0x7fc00000);
    }
}

// Shared memory of the extra token's draw.
struct DrawSmem {
    unsigned long long span_total;
    unsigned long long tau, W, base;
    int owner, mode, tile;
    // pushed span totals: slot r from CTA r, completing on tbar
    unsigned long long totals[kSeqMaxCluster];
    uint64_t tbar;
};

// The extra token of sequence b (Appendix A.1; reading 4 and 4b for the
// convention and the arithmetic): inverse CDF of w = max(0, p_a - q_a) when
// a < k, of p_k when a = k.  This CTA, rank `rank` of a cluster of p.csize,
// owns entries [e0, e0 + n) of the vocabulary: it sums their weights per
// sub-tile (fp32 in a warp, exact 64-bit fixed point beyond), the CTAs' span
// totals meet through distributed shared memory, and the CTA whose span holds
// tau = floor(u W) rescans that one sub-tile exactly.  Entry j of the target and
// draft rows at position a is trow[j - off], zrow[j - off]; kMode says in which
// memory and how aligned.  trow_g is the whole target row in global memory, for the
// case W = 0 (argmax of p_a).  s_sub holds at least n / (32 kVec) floats.  Every thread
// calls it.  Each CTA pushes its total by st.async into slot `rank` of every
// CTA's ds.totals and waits on its own ds.tbar (initialised with count 1 and visible
// to the cluster): no cluster barrier, nothing read from a peer.  Returns false if
// that wait gave up (the draw is then not made).
template <typename In, int kMode, int kThreads>
__device__ __forceinline__ bool residual_draw(const FinParams& p, int b, int a, const SeqSmem& sh, int rank,
                                              int e0, int n, const In* trow, const In* zrow, int off,
                                              const In* trow_g, float* s_sub, DrawSmem& ds) {
    using E = Elem<In>;
    constexpr int kW = E::kVec;  // entries per lane per sub-tile
    constexpr int kSub = 32 * kW;
    constexpr int kWarps = kThreads / 32;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int k = p.k, V = p.V;
    const bool bonus = (a == k);
    int32_t* out = p.out_tokens + size_t(b) * (k + 1);
    // kW entries from entry j of a row, and one entry; `whole`: all kW belong to this span
    auto ldv = [&](const In* row, int j) {
        if constexpr (kMode == kRowsStaged) return lds_v4(row + (j - off));
        else if constexpr (kMode == kRowsAligned) return ldg_stream(row + (j - off));
        else return ldg_shifted(row + (j - off));
    };
    auto ld1 = [&](const In* row, int j) {
        return kMode == kRowsStaged ? E::lds(row + (j - off)) : E::load(row + (j - off));
    };
    // unaligned rows: the aligned vectors around the entries have to lie within the row
    auto inside = [&](const In* row, int j) {
        if constexpr (kMode != kRowsAny) return true;
        else return shifted_inside(row, j, V);
    };
    const float mt = sh.m[a], inv_st = 1.0f / sh.s[a];
    const float mz = bonus ? 0.f : sh.m[k + 1 + a];
    const float st_sz = bonus ? 0.f : sh.s[a] / sh.s[k + 1 + a];
    const float ch = p.c_hi, cl = p.c_lo;
    const int nsub = (n + kSub - 1) / kSub;  // sub-tiles: one warp step of 32 x kW entries
    // raw entries of this lane in sub-tile s (slots past the span read as -inf: weight 0)
    struct Raw {
        uint4 t, z;
    };
    auto load_sub = [&](auto has_q, int s, Raw& r) {
        constexpr bool kQ = decltype(has_q)::value;
        const int j0 = e0 + s * kSub + lane * kW;
        const int cnt = min(kW, e0 + n - j0);
        if (cnt == kW && inside(trow, j0) && (!kQ || inside(zrow, j0))) {
            r.t = ldv(trow, j0);
            if constexpr (kQ) r.z = ldv(zrow, j0);
        } else {
            float tv[kW], zv[kW];
#pragma unroll
            for (int e = 0; e < kW; ++e) {
                tv[e] = (e < cnt) ? ld1(trow, j0 + e) : kNegInf;
                zv[e] = (e < cnt && kQ) ? ld1(zrow, j0 + e) : kNegInf;
            }
            r.t = pack_raw<In, kW>(tv);
            if constexpr (kQ) r.z = pack_raw<In, kW>(zv);
        }
    };
    // residual weights of one sub-tile slot times st, the target row's sum, in pairs:
    // e_t, or max(0, e_t - e_z st / sz) with one rounding, so that entries of equal
    // probability weigh exactly 0 where the two sums are equal.  (The difference of two
    // rounded products does not: ptxas fuses a packed product into it.)  has_q (a
    // std::true_type) unless a = k: with a branch on `bonus` among the loads and sums instead, B =
    // 256, k = 8, V = 128256 took 78.8 us where it takes 69.9 (0.13 accepted), k = 1 71.1 for 63.9.
    auto sub_weights = [&](auto has_q, const Raw& r, float2* w) {
        float2 d[kW / 2];
        E::minus(r.t, mt, d);
#pragma unroll
        for (int e = 0; e < kW / 2; ++e) w[e] = exp2_pair(d[e], ch, cl);
        if constexpr (decltype(has_q)::value) {
            E::minus(r.z, mz, d);
#pragma unroll
            for (int e = 0; e < kW / 2; ++e) {
                const float2 df = fma2(exp2_pair(d[e], ch, cl), f2(-st_sz), w[e]);
                w[e] = make_float2(fmaxf(df.x, 0.f), fmaxf(df.y, 0.f));
            }
        }
    };

    // pass 1: one fp32 sum per sub-tile, no block barrier; the sums of a step are
    // reduced over the lanes together
    static_assert(kFinUnroll == 4, "warp_sum4 carries four sums");
    auto pass1 = [&](auto has_q) {
        for (int s0 = warp; s0 < nsub; s0 += kWarps * kFinUnroll) {
            Raw r[kFinUnroll];
#pragma unroll
            for (int u = 0; u < kFinUnroll; ++u)
                if (s0 + u * kWarps < nsub) load_sub(has_q, s0 + u * kWarps, r[u]);
            float sum[kFinUnroll];
#pragma unroll
            for (int u = 0; u < kFinUnroll; ++u) {
                sum[u] = 0.f;
                if (s0 + u * kWarps < nsub) {
                    float2 w[kW / 2];
                    sub_weights(has_q, r[u], w);
                    float2 s2 = w[0];
#pragma unroll
                    for (int e = 1; e < kW / 2; ++e) s2 = add2(s2, w[e]);
                    sum[u] = s2.x + s2.y;
                }
            }
            const float tot = warp_sum4(sum);
            const int s = s0 + (lane >> 3) * kWarps;
            if ((lane & 7) == 0 && s < nsub) s_sub[s] = tot * inv_st;
        }
    };
    if (bonus) pass1(std::false_type());
    else pass1(std::true_type());
    __syncthreads();
    // span total, exact, reduced across warp 0
    bool got = true;
    if (warp == 0) {
        unsigned long long part = 0ull;
        for (int s2 = lane; s2 < nsub; s2 += 32) part += fix_of(s_sub[s2]);
        part = warp_sum_u64(part);
        if (lane == 0) ds.span_total = part;
        if (p.csize > 1) {
            if (lane < p.csize)
                st_async_u64(map_rank(&ds.totals[rank], static_cast<uint32_t>(lane)), part,
                             map_rank(&ds.tbar, static_cast<uint32_t>(lane)));
            if (lane == 0) mbar_arrive_expect_tx(&ds.tbar, static_cast<uint32_t>(p.csize) * 8u);
            got = __all_sync(0xffffffffu, mbar_wait_cluster_bounded(&ds.tbar, 0, kPeerWaitNs));
        }
    }
    __syncthreads();

    // warp 0 of every CTA derives W, tau = floor(u W) and the owning CTA identically:
    // lane r holds CTA r's total, a warp scan gives the prefix in rank order
    if (warp == 0 && got) {
        const float u = sh.u[k];
        unsigned long long tot = 0ull;
        if (lane < p.csize) tot = (p.csize > 1) ? ds.totals[lane] : ds.span_total;
        const unsigned long long incl = warp_incl_scan_u64(tot);
        const unsigned long long W = __shfl_sync(0xffffffffu, incl, 31);
        const unsigned long long tau = fix_scale(u, W);
        int owner, mode = 0;  // mode 0: inverse CDF, 1: largest positive entry, 2: argmax p
        unsigned long long base = 0ull;
        if (W > 0ull) {
            const unsigned hit = __ballot_sync(0xffffffffu, lane < p.csize && incl > tau);
            if (hit) {
                owner = __ffs(hit) - 1;
                base = __shfl_sync(0xffffffffu, incl - tot, owner);
            } else {  // tau >= W (u >= 1 or rounding): largest j with w_j > 0
                mode = 1;
                const unsigned pos = __ballot_sync(0xffffffffu, lane < p.csize && tot > 0ull);
                owner = 31 - __clz(pos);
            }
        } else {
            mode = 2;
            owner = 0;
        }
        int tile = -1;
        if (rank == owner) {
            // sub-tile holding tau: each lane owns a run of consecutive sub-tiles
            const int per = (nsub + 31) / 32;
            const int s_lo = min(nsub, lane * per), s_hi = min(nsub, s_lo + per);
            unsigned long long mine = 0ull;
            for (int s2 = s_lo; s2 < s_hi; ++s2) mine += fix_of(s_sub[s2]);
            const unsigned long long excl = base + warp_incl_scan_u64(mine) - mine;
            if (mode == 0) {
                const unsigned hit = __ballot_sync(0xffffffffu, excl <= tau && excl + mine > tau);
                if (hit) {
                    const int l = __ffs(hit) - 1;
                    if (lane == l) {  // the sums are exact: the run holds tau in one sub-tile
                        unsigned long long c = excl;
                        for (int s2 = s_lo; s2 < s_hi; ++s2) {
                            const unsigned long long v = fix_of(s_sub[s2]);
                            if (c + v > tau) { tile = s2; break; }
                            c += v;
                        }
                        base = c;
                    }
                    tile = __shfl_sync(0xffffffffu, tile, l);
                    base = __shfl_sync(0xffffffffu, base, l);
                } else {
                    mode = 1;
                }
            }
            if (mode == 1) {  // the last sub-tile with positive mass
                int last = -1;
                for (int s2 = s_lo; s2 < s_hi; ++s2)
                    if (s_sub[s2] > 0.f) last = s2;
                for (int o = 16; o > 0; o >>= 1) last = max(last, __shfl_xor_sync(0xffffffffu, last, o));
                tile = last;
            }
        }
        if (lane == 0) { ds.owner = owner; ds.mode = mode; ds.tau = tau; ds.W = W; ds.base = base; ds.tile = tile; }
    }
    if (warp == 0 && lane == 0 && !got) ds.owner = -1;
    __syncthreads();
    if (ds.owner < 0) return false;

    if (rank == ds.owner && warp == 0) {
        const unsigned long long tau = ds.tau, W = ds.W;
        const int mode = ds.mode, s = ds.tile;
        if (mode == 0 || mode == 1) {
            float w[kW];
            {
                float2 w2[kW / 2];
                auto at_tile = [&](auto has_q) {
                    Raw r;
                    if (s >= 0) load_sub(has_q, s, r);
                    else { r.t = ninf_raw<In>(); r.z = r.t; }
                    sub_weights(has_q, r, w2);
                };
                if (bonus) at_tile(std::false_type());
                else at_tile(std::true_type());
#pragma unroll
                for (int e = 0; e < kW / 2; ++e) {
                    w[2 * e] = w2[e].x * inv_st;
                    w[2 * e + 1] = w2[e].y * inv_st;
                }
            }
            const int j0 = e0 + max(s, 0) * kSub + lane * kW;
            bool done = false;
            if (mode == 0) {
                // exact scan of the sub-tile across the warp, then within the lane
                unsigned long long mine = 0ull;
#pragma unroll
                for (int e = 0; e < kW; ++e) mine += fix_of(w[e]);
                const unsigned long long excl = ds.base + warp_incl_scan_u64(mine) - mine;
                const bool hit = excl <= tau && excl + mine > tau;
                if (hit) {
                    unsigned long long C = excl;
                    for (int e = 0; e < kW; ++e) {
                        const unsigned long long Cprev = C;
                        C += fix_of(w[e]);
                        if (C > tau) {
                            out[a] = j0 + e;
                            if (p.diag_gap)
                                p.diag_gap[b] = fminf(fix_to_float(C - tau), fix_to_float(tau - Cprev)) / fix_to_float(W);
                            break;
                        }
                    }
                }
                done = __any_sync(0xffffffffu, hit);
            }
            if (!done) {
                // largest j of the sub-tile with w_j > 0 (rounding fallback)
                int best = -1;
                float wbest = 0.f;
#pragma unroll
                for (int e = 0; e < kW; ++e)
                    if (w[e] > 0.f) { best = j0 + e; wbest = w[e]; }
                int jb = best;
                for (int o = 16; o > 0; o >>= 1) jb = max(jb, __shfl_xor_sync(0xffffffffu, jb, o));
                if (jb >= 0 && best == jb) {
                    out[a] = jb;
                    if (p.diag_gap) {
                        const float Wf = fix_to_float(W), tf = fix_to_float(tau);
                        p.diag_gap[b] = fminf(Wf - tf, tf - (Wf - wbest)) / Wf;
                    }
                } else if (jb < 0 && lane == 0) {
                    out[a] = e0;  // no positive entry found: cannot happen when W > 0
                }
            }
        } else {
            // no residual mass at all: argmax of p_a over the whole row
            MaxIdx acc{kNegInf, INT_MAX};
            for (int j = lane; j < V; j += 32) {
                const float t = E::load(trow_g + j);
                if (t > acc.m) { acc.m = t; acc.i = j; }
            }
            acc = warp_reduce(acc, [](MaxIdx x, MaxIdx y) { return merge_mi(x, y); });
            if (lane == 0) {
                out[a] = (acc.i == INT_MAX) ? 0 : acc.i;
                if (p.diag_gap) p.diag_gap[b] = __int_as_float(0x7fc00000);
            }
        }
    }
    return true;
}

// ------------------------------------------------------------------ rows on demand (T > 0)
// The tests run in order and nothing past the first failure is decided, so the
// rows past it are never needed.  One thread-block cluster per sequence walks the
// positions in rounds: its CTAs, each owning a span of the vocabulary, stream the
// round's rows once (warps shared out over the rows), exchange the span statistics
// by st.async, and every CTA merges the same slots in rank order and runs the
// round's accept tests, so all decide alike without a further exchange.  An
// accepted round doubles the next one's positions.  At the first failure (or after
// the bonus row) the cluster draws the extra token from rows that L2 mostly still
// holds.
//
// What bounds it: with a poor draft at B = 256, k = 8, V = 128256 (0.13 accepted) the two
// rows a sequence needs are 148 MB, 22 us at the copy bandwidth; it takes 70 us (all
// rows in two launches: 211 us), half of the issue slots idle while the dependent phases
// (statistics, exchange, draw) wait for each other.  The same batch with 3.0 accepted takes
// 148 us (211), with 5.6 185 us (209), with 7.1, where nearly every row is read, 209 us (208).
// 64 registers and four CTAs an SM with groups of 4 vectors in flight measured best, at 76 us
// (groups of 2 with five or six CTAs: 84 us); staging the first position in shared memory
// at these sizes, three CTAs an SM, then gave 70 us with the poor draft and 257 us with the good
// one, whose rounds wait for their copies.
constexpr int kLazyMaxWin = 8;                 // positions per round ...
constexpr int kLazyMaxRows = 2 * kLazyMaxWin;  // ... two rows each
constexpr int kLazyThreads = 256;
constexpr int kStagedThreads = 512;          // with a staged first round: one CTA an SM

// Byte offset of the sub-tile sums in the kernel's dynamic shared memory: after the
// staged rows of the first round (none when kStaged is off).
__host__ __device__ inline size_t lazy_sub_offset(int nslots, int span, size_t es) {
    return (size_t(nslots) * span * es + 15) / 16 * 16;
}

// kStaged (16-byte-aligned rows): the first round's rows are bulk-copied to shared memory,
// and a draw at one of its positions, the usual one with a draft that is often wrong,
// reads them there.
template <typename In, bool kStaged, bool kAligned>
__global__ void __launch_bounds__(kStaged ? kStagedThreads : kLazyThreads, kStaged ? 1 : 4)
verify_lazy_kernel(FinParams p, int win, int ahead) {
    static_assert(kAligned || !kStaged, "bulk copies want 16-byte-aligned rows");
    using E = Elem<In>;
    constexpr int kVec = E::kVec;
    constexpr int kThreads = kStaged ? kStagedThreads : kLazyThreads, kWarps = kThreads / 32;
    __shared__ SeqSmem sh;
    __shared__ DrawSmem ds;
    __shared__ MaxSum s_part[kWarps > kLazyMaxRows ? kWarps : kLazyMaxRows];
    __shared__ __align__(8) MaxSum s_recv[2][kSeqMaxCluster * kLazyMaxRows];  // [CTA][row], two rounds
    __shared__ __align__(8) uint64_t s_bar[2];
    __shared__ __align__(8) uint64_t s_rbar[kLazyMaxRows];  // staged rows
    __shared__ int s_dec;  // first failing position, k after the bonus row, -1 undecided, -2 a wait gave up
    extern __shared__ __align__(128) unsigned char lsm[];

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int csize = p.csize;
    const int rank = (csize > 1) ? static_cast<int>(cluster_rank()) : 0;
    const int b = blockIdx.x / csize;
    const int k = p.k, V = p.V;
    const int e0 = rank * p.span;
    const int n = min(p.span, V - e0);
    const In* draft = static_cast<const In*>(p.draft) + size_t(b) * k * V;
    const In* target = static_cast<const In*>(p.target) + size_t(b) * (k + 1) * V;
    const float ch = p.c_hi, cl = p.c_lo;
    In* staged = reinterpret_cast<In*>(lsm);
    float* s_sub = reinterpret_cast<float*>(lsm + (kStaged ? lazy_sub_offset(min(2 * win, 2 * p.k + 1), p.span, sizeof(In)) : 0));
    const int w0 = min(win, k + 1);  // positions of the first round
    // row q of the round of w positions from i0: the target rows first, then the draft rows
    // (the bonus position k has none)
    auto row_of = [&](int i0, int w, int q) {
        return ((q < w) ? target + size_t(i0 + q) * V : draft + size_t(i0 + q - w) * V) + e0;
    };
    auto rows_of = [&](int i0, int w) { return 2 * w - (i0 + w == k + 1 ? 1 : 0); };

    if (tid == 0) {
        mbar_init_only(&s_bar[0], 1);
        mbar_init_only(&s_bar[1], 1);
        mbar_init_only(&ds.tbar, 1);
        if constexpr (kStaged)
            for (int q = 0; q < kLazyMaxRows; ++q) mbar_init_only(&s_rbar[q], 1);
        fence_mbarrier_init();
    }
    grid_dependency_sync();
    if constexpr (kStaged) {
        if (tid == 0) {
            const uint32_t bytes = static_cast<uint32_t>(n * sizeof(In));  // a multiple of 16 on this path
            for (int q = 0; q < rows_of(0, w0); ++q) {
                mbar_arrive_expect_tx(&s_rbar[q], bytes);
                bulk_g2s(staged + size_t(q) * p.span, row_of(0, w0, q), bytes, &s_rbar[q]);
            }
            if (ahead && w0 <= k) {  // the second round's rows start on their way to L2
                const int w1 = min(min(2 * w0, kLazyMaxWin), k + 1 - w0);
                for (int q = 0; q < rows_of(w0, w1); ++q) bulk_prefetch_l2(row_of(w0, w1, q), bytes);
            }
        }
    }
    __syncthreads();  // the barriers are initialised before anyone waits on them
    // ... and before any peer pushes to them: arrive now, wait before the first push
    if (csize > 1) cluster_arrive_relaxed();
    // the draft tokens, the two logits each accept test needs, and the uniforms: two dependent
    // loads of one warp, which the others do not wait for before they start on the rows
    int bad = 0;
    if (warp == kWarps - 1) {
        const int32_t* y = p.tokens + size_t(b) * k;
        for (int i = lane; i < k; i += 32) {
            const int t = y[i];
            sh.y[i] = t;
            if (t < 0 || t >= V) {
                bad = 1;
            } else {
                sh.zy[i] = E::load(draft + size_t(i) * V + t);
                sh.ty[i] = E::load(target + size_t(i) * V + t);
            }
        }
    }
    if (warp == kWarps - 2)
        for (int i = lane; i <= k; i += 32) sh.u[i] = p.uniforms[size_t(b) * (k + 1) + i];

    int a = -1, i0 = 0, w = w0;
    unsigned round = 0;
    bool stuck = false;  // a staging copy gave up in this CTA
    for (;;) {
        const int nr = rows_of(i0, w);
        const int parts = max(1, kWarps / nr);  // warps per row: all kWarps on a lone bonus row
        int timed_out = 0;
        for (int it = warp; it < nr * parts; it += kWarps) {
            const int q = it / parts, part = it - q * parts;
            MaxSum mine;
            if (kStaged && round == 0) {
                if (!mbar_wait_bounded(&s_rbar[q], 0, kStageWaitNs)) timed_out = 1;
                const int nch = n / kVec;
                mine = staged_stats<In>(staged + size_t(q) * p.span, nch * part / parts, nch * (part + 1) / parts, ch, cl);
            } else {
                mine = span_stats<In>(row_of(i0, w, q), n, part, parts, ch, cl);
            }
            if (lane == 0) s_part[it] = mine;
        }
        if (round == 0) {
            if (__syncthreads_or(timed_out | bad)) {
                if constexpr (kStaged)  // every copy lands, or gets a last chance to, before this CTA goes on or leaves
                    for (int q = 0; q < nr; ++q) mbar_wait_bounded(&s_rbar[q], 0, kStageWaitNs);
                if (__syncthreads_or(bad)) {  // uniform over the cluster, before any push to a peer
                    if (rank == 0) seq_write_bad<kThreads>(p, b);
                    return;
                }
                stuck = true;
            }
            if (csize > 1) asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
        } else {
            __syncthreads();
        }
        if (warp == 0) {
            const int dec = seq_round<kWarps>(p, b, sh, s_part, parts, s_recv[round & 1u], kLazyMaxRows, &s_bar[round & 1u],
                                              (round >> 1) & 1u, rank, i0, w, nr, stuck);
            if (lane == 0) s_dec = dec;
        }
        __syncthreads();
        a = s_dec;
        if (a != -1) break;
        // an accepted round makes a longer one likely to pass: twice the positions
        i0 += w;
        w = min(min(2 * w, kLazyMaxWin), k + 1 - i0);
        ++round;
    }
    if (a < 0) {  // a row or the peers' statistics did not arrive in time: the sequence is reported as bad
        if (csize > 1 && tid == 0) mbar_wait_cluster_bounded(&s_bar[round & 1u], (round >> 1) & 1u, kPeerWaitNs);
        if (rank == 0) seq_write_bad<kThreads>(p, b);
        return;
    }
    if (rank == 0) seq_write_outputs<kThreads>(p, b, sh, a);
    const In* trow = target + size_t(a) * V;
    const In* zrow = draft + size_t(a == k ? 0 : a) * V;
    bool drawn;
    if (kStaged && a < w0)
        drawn = residual_draw<In, kRowsStaged, kThreads>(p, b, a, sh, rank, e0, n, staged + size_t(a) * p.span,
                                                         staged + size_t(a == k ? a : w0 + a) * p.span, e0, trow, s_sub, ds);
    else
        drawn = residual_draw<In, kAligned ? kRowsAligned : kRowsAny, kThreads>(p, b, a, sh, rank, e0, n, trow, zrow, 0,
                                                                                trow, s_sub, ds);
    if (!drawn) seq_write_bad<kThreads>(p, b);
}

// ------------------------------------------------------------------ every row staged (T > 0)
// At serving batch sizes one round of latency costs more than the bytes of rows that
// turn out not to be needed: each CTA of the sequence's cluster bulk-copies its
// vocabulary span of all 2k + 1 rows (all the copies in flight at once, a barrier
// per row, so that a row's statistics start as soon as it has landed), and one
// exchange decides all the positions.  It runs only when its grid fits in one wave with
// slots to spare (see launch_sampling).  At B = 32, k = 5, V = 32000 (22 MB, 3.3 us at the copy
// bandwidth) it takes 11.4 us back to back, 19.0 us alone with a cold L2: a chain of copy,
// statistics, exchange, tests and draw.  512 threads (256 threads 12 % more; 16-CTA
// clusters 60 % more).
constexpr int kFuseThreads = 512;
constexpr int kFuseParts = 4;           // warp items per row for the span statistics
constexpr int kFuseMaxB = 64;           // at most this many sequences, and the grid in one wave

// Byte offset of the receive slots in the dynamic shared memory: after the staged
// rows and the sub-tile sums, 16-byte aligned.
__host__ __device__ inline size_t fused_recv_offset(int nrows, int span, size_t es) {
    return (size_t(nrows) * span * es + size_t(span / 128 + 1) * sizeof(float) + 15) / 16 * 16;
}

template <typename In>
__global__ void __launch_bounds__(kFuseThreads) verify_fused_kernel(FinParams p) {
    using E = Elem<In>;
    constexpr int kVec = E::kVec;
    constexpr int kWarps = kFuseThreads / 32;
    constexpr int kMaxRows = 2 * OSD_VERIFY_MAX_K + 1;
    extern __shared__ __align__(128) unsigned char fsm[];
    __shared__ __align__(8) uint64_t rbar[kMaxRows];  // one staging barrier per row
    __shared__ SeqSmem sh;
    __shared__ DrawSmem ds;
    __shared__ MaxSum s_part[kMaxRows * kFuseParts];
    __shared__ __align__(8) uint64_t s_bar;  // the cluster's span statistics have arrived
    __shared__ int s_dec;  // as in verify_lazy_kernel

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int csize = p.csize;
    const int rank = (csize > 1) ? static_cast<int>(cluster_rank()) : 0;
    const int b = blockIdx.x / csize;
    const int k = p.k, V = p.V;
    const int nrows = 2 * k + 1;
    const int e0 = rank * p.span;
    const int n = min(p.span, V - e0);
    const In* draft = static_cast<const In*>(p.draft) + size_t(b) * k * V;
    const In* target = static_cast<const In*>(p.target) + size_t(b) * (k + 1) * V;
    In* rows = reinterpret_cast<In*>(fsm);  // row q <= k is target row q, q > k draft row q - k - 1
    float* s_sub = reinterpret_cast<float*>(fsm + size_t(nrows) * p.span * sizeof(In));
    // [csize][nrows]: CTA c's span statistics of every row, pushed by CTA c
    MaxSum* recv = reinterpret_cast<MaxSum*>(fsm + fused_recv_offset(nrows, p.span, sizeof(In)));
    const uint32_t bytes = static_cast<uint32_t>(n * sizeof(In));  // a multiple of 16 on this path

    if (tid == 0) {
        for (int q = 0; q < nrows; ++q) mbar_init_only(&rbar[q], 1);
        mbar_init_only(&s_bar, 1);
        mbar_init_only(&ds.tbar, 1);
        fence_mbarrier_init();
    }
    grid_dependency_sync();
    if (tid == 0) {
        for (int q = 0; q < nrows; ++q) {
            mbar_arrive_expect_tx(&rbar[q], bytes);
            bulk_g2s(rows + size_t(q) * p.span,
                     ((q <= k) ? target + size_t(q) * V : draft + size_t(q - k - 1) * V) + e0, bytes, &rbar[q]);
        }
    }
    __syncthreads();  // the barriers are initialised before anyone waits on them
    // ... and before any peer pushes to them: arrive now, wait before the first push
    if (csize > 1) cluster_arrive_relaxed();
    // meanwhile the draft tokens, the two logits each accept test needs, and the uniforms
    int bad = 0;
    if (warp == kWarps - 1) {
        const int32_t* y = p.tokens + size_t(b) * k;
        for (int i = lane; i < k; i += 32) {
            const int t = y[i];
            sh.y[i] = t;
            if (t < 0 || t >= V) {
                bad = 1;
            } else {
                sh.zy[i] = E::load(draft + size_t(i) * V + t);
                sh.ty[i] = E::load(target + size_t(i) * V + t);
            }
        }
    }
    if (warp == kWarps - 2)
        for (int i = lane; i <= k; i += 32) sh.u[i] = p.uniforms[size_t(b) * (k + 1) + i];

    // span statistics of every row: warp items (row, part)
    const int nch = n / kVec;
    int timed_out = 0;
    for (int it = warp; it < nrows * kFuseParts; it += kWarps) {
        const int q = it / kFuseParts, part = it - q * kFuseParts;
        if (!mbar_wait_bounded(&rbar[q], 0, kStageWaitNs)) timed_out = 1;
        const MaxSum mine = staged_stats<In>(rows + size_t(q) * p.span, nch * part / kFuseParts,
                                             nch * (part + 1) / kFuseParts, p.c_hi, p.c_lo);
        if (lane == 0) s_part[it] = mine;
    }
    bool stuck = false;
    if (__syncthreads_or(timed_out | bad)) {
        // every copy lands, or gets a last chance to, before this CTA goes on or leaves
        for (int q = 0; q < nrows; ++q) mbar_wait_bounded(&rbar[q], 0, kStageWaitNs);
        if (__syncthreads_or(bad)) {  // uniform over the cluster, before any push to a peer
            if (rank == 0) seq_write_bad<kFuseThreads>(p, b);
            return;
        }
        stuck = true;
    }
    if (csize > 1) asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    if (warp == 0) {
        const int dec =
            seq_round<kFuseParts>(p, b, sh, s_part, kFuseParts, recv, nrows, &s_bar, 0, rank, 0, k + 1, nrows, stuck);
        if (lane == 0) s_dec = dec;
    }
    __syncthreads();
    const int a = s_dec;
    if (a < 0) {  // the GPU did not deliver a row in time: the sequence is reported as bad
        if (csize > 1 && tid == 0) mbar_wait_cluster_bounded(&s_bar, 0, kPeerWaitNs);
        if (rank == 0) seq_write_bad<kFuseThreads>(p, b);
        return;
    }
    if (rank == 0) seq_write_outputs<kFuseThreads>(p, b, sh, a);
    // ---- extra token from the staged rows at position a
    const In* trow_s = rows + size_t(a) * p.span;
    const In* zrow_s = (a == k) ? trow_s : rows + size_t(k + 1 + a) * p.span;
    // (a peer whose pushed total did not arrive in time reports the sequence as bad)
    if (!residual_draw<In, kRowsStaged, kFuseThreads>(p, b, a, sh, rank, e0, n, trow_s, zrow_s, e0,
                                                      target + size_t(a) * V, s_sub, ds))
        seq_write_bad<kFuseThreads>(p, b);
}

// ------------------------------------------------------------------ host
static int verify_slice_len(int B, int k) { return stats_slice_len((long long)B * (2 * k + 1)); }

static int verify_slices(int B, int k, int V) {
    const int len = verify_slice_len(B, k);
    return (V + len - 1) / len;
}

static size_t round256(size_t x) { return (x + 255) / 256 * 256; }

// Split V over at most c CTAs in spans of a multiple of 64 entries.
static void split_vocab(int V, int c, FinParams* fp) {
    int s = (V + c - 1) / c;
    s = (s + 63) / 64 * 64;
    fp->span = s;
    fp->csize = (V + s - 1) / s;
}

// T > 0: which kernel, CTAs per sequence and positions per round.
template <typename In>
static osd_status launch_sampling(FinParams fp, cudaStream_t stream) {
    const int B = fp.B, k = fp.k, V = fp.V;
    constexpr size_t es = sizeof(In);
    const bool aligned = aligned_to(fp.target, 16) && aligned_to(fp.draft, 16) && ((size_t)V * es) % 16 == 0;
    if (aligned && B <= kFuseMaxB) {
        // every row staged, only in one wave and with slots to spare, since a grid that just
        // fits finds them scattered over the GPCs: at B = 32, k = 5, V = 32000 (two CTAs an SM, 256
        // of 304 slots) 11.4 us whatever the draft, against 13.3 us on demand from 2 accepted on (11.6
        // with 0.6); at B = 36, V = 20224 (288) 14.2 against 12.0
        split_vocab(V, kSeqMaxCluster, &fp);
        const size_t smem = fused_recv_offset(2 * k + 1, fp.span, es) + size_t(fp.csize) * (2 * k + 1) * sizeof(MaxSum);
        if (smem <= kStageMaxSmem &&
            (long long)B * fp.csize * 8 <= (long long)device_sms() * ctas_per_sm<verify_fused_kernel<In>, kFuseThreads>(smem) * 7)
            return from_cuda(launch_ex(true, verify_fused_kernel<In>, dim3(unsigned(B) * unsigned(fp.csize)), dim3(kFuseThreads),
                                    smem, stream, fp.csize, fp));
    }
    // Rows on demand.  A round costs about 2 us beside its bytes, and positions past the
    // first failure are read for nothing: the first round takes 1 position from 40 MB a position
    // of the batch on (B = 233, k = 4, V = 27472 fp32, 51 MB: 42.3 us against 44.5 and 45.0 with 2 and
    // 4), 2 from 10 MB (B = 204, k = 4, V = 14144 fp32, 23 MB: 26.1, level with 26.5 and 25.5 with 1 and
    // 4), 4 from 2 MB (B = 100, k = 4, V = 23488, 9 MB: 17.5 against 18.2 and 20.4 with 2 and 1; at
    // B = 51, k = 6, V = 10944, 2.2 MB, 8 would do better, 10.7 against 12.6), else 8.
    constexpr int sub = 32 * Elem<In>::kVec;
    auto sub_bytes = [&]() { return size_t((fp.span + sub - 1) / sub) * sizeof(float); };
    const double pos = double(B) * 2 * V * double(es);  // bytes of one position of the batch
    const int win = pos > 40e6 ? 1 : (pos > 10e6 ? 2 : (pos > 2e6 ? 4 : kLazyMaxWin));
    const int most = std::max(1, std::min<int>(kSeqMaxCluster, int(size_t(V) * es / 2048)));  // spans of 2 KB or more
    if (aligned && B <= device_sms() / 2) {
        // the first round staged where the batch runs at one CTA an SM, with fewer positions
        // where they do not fit (B = 16, k = 8, V = 128256, 2 positions: 27.7 us against 43.7 us streamed;
        // B = 36, k = 6, V = 20224: level, 12.6 us), in pairs of SMs: with clusters of 3 or 5 a batch
        // that just fits is slower (B = 28, k = 5, V = 8704, 5 CTAs: 13.8 us, 4: 8.7)
        const int c = widest_cluster<verify_lazy_kernel<In, true, true>, kStagedThreads>(B, most, kStageMaxSmem, false) & ~1;
        if (c >= 2) split_vocab(V, c, &fp);
        for (int w = win; w >= 1 && c >= 2; w /= 2) {
            const size_t smem = lazy_sub_offset(std::min(2 * w, 2 * k + 1), fp.span, es) + sub_bytes();
            if (smem <= kStageMaxSmem && ctas_per_sm<verify_lazy_kernel<In, true, true>, kStagedThreads>(smem) >= 1) {
                // so small a second round that its bytes cost nothing if the first one rejects
                const int ahead = pos * std::min(2 * w, kLazyMaxWin) <= 9e6;
                return from_cuda(launch_ex(true, verify_lazy_kernel<In, true, true>, dim3(unsigned(B) * unsigned(fp.csize)),
                                        dim3(kStagedThreads), smem, stream, fp.csize, fp, w, ahead));
            }
            if (c == 2) break;  // long spans: streamed at four CTAs an SM instead
        }
    }
    // one wave of the widest clusters, not quite full, since a grid that just fits waits for its last
    // slots (B = 192, k = 4, V = 11200 with 3 CTAs a sequence, of which 194 fit: 20.9 us, with 2 18.3;
    // B = 84, k = 4, V = 38180 fp32, 6 CTAs: 26.8 us, with 8, of which 74 fit, 31.5; B = 186, k = 2, V = 24576,
    // 3: 18.0, with 4 23.2), as long as L2 holds a position for the draw; past that the fewest CTAs
    // whose spans stay within 68 KB, so that the rows in flight do (B = 256, k = 8, V = 128256 8 CTAs,
    // 70 us against 77 and 95 us with 4 and 2)
    int c = most;
    if (pos <= 100e6) {
        // (batches past one wave: B = 340, k = 4, 2 CTAs against 1: V = 32000 46.3 and 58.7 us, V = 8192
        // 23.6 and 22.1)
        const int c1 = size_t(V) * es >= 48 * 1024 ? 2 : 1;
        // the sub-tile sums of any span here: of V <= 2^21 fp32 entries over 8 CTAs 8 KB, over fewer
        // (then the batch is larger and, within 100 MB, V smaller) less
        constexpr size_t kSubs = 8192;
        c = std::max(c1, aligned ? widest_cluster<verify_lazy_kernel<In, false, true>, kLazyThreads>(B, most, kSubs, true)
                                : widest_cluster<verify_lazy_kernel<In, false, false>, kLazyThreads>(B, most, kSubs, true));
    } else {
        while (c > 1 && size_t(V / (c / 2)) * 2 * es <= 68 * 1024) c /= 2;
    }
    split_vocab(V, c, &fp);
    if ((long long)B * fp.csize > INT_MAX) return OSD_ERR_UNSUPPORTED;
    const dim3 grid(unsigned(B) * unsigned(fp.csize));
    return from_cuda(aligned ? launch_ex(true, verify_lazy_kernel<In, false, true>, grid, dim3(kLazyThreads), sub_bytes(), stream,
                                      fp.csize, fp, win, 0)
                             : launch_ex(true, verify_lazy_kernel<In, false, false>, grid, dim3(kLazyThreads), sub_bytes(), stream,
                                      fp.csize, fp, win, 0));
}

template <typename In>
static osd_status launch_verify(const void* draft, const void* target, int B, int k, int V,
                                const int32_t* tokens, const float* uniforms, float T,
                                int32_t* accepted, int32_t* out_tokens, uint8_t* mask,
                                float* diag_margin, float* diag_gap, RowStat* stats,
                                cudaStream_t stream) {
    const bool greedy = (T == 0.f);
    FinParams fp = {};
    fp.draft = draft; fp.target = target; fp.B = B; fp.k = k; fp.V = V;
    fp.tokens = tokens; fp.uniforms = uniforms; fp.T = T;
    fp.accepted = accepted; fp.out_tokens = out_tokens; fp.mask = mask;
    fp.diag_margin = diag_margin; fp.diag_gap = diag_gap;
    if (greedy) {
        osd_status st = OSD_OK;
        if (launch_greedy_walk<In>(GreedyChain{fp}, static_cast<const In*>(target), B, k + 1, k + 1, V, stream, &st)) return st;
        const int slice_len = verify_slice_len(B, k);
        fp.n_slices = verify_slices(B, k, V);
        fp.stats = stats;
        const long long grid1 = (long long)B * (k + 1) * fp.n_slices;
        if (grid1 > INT_MAX) return OSD_ERR_UNSUPPORTED;
        const cudaError_t e =
            launch_ex(true, row_argmax_kernel<In>, dim3(unsigned(grid1)), dim3(kStatThreads), 0, stream, 1,
                   static_cast<const In*>(target), V, slice_len, fp.n_slices, stats);
        if (e != cudaSuccess) return OSD_ERR_CUDA;
        fp.csize = 1;
        fp.span = V;
        const dim3 grid_g(unsigned((B + kGreedyWarps - 1) / kGreedyWarps));
        return from_cuda(launch_ex(true, verify_greedy_kernel, grid_g, dim3(kGreedyWarps * 32), 0, stream, 1, fp));
    }
    split_scale(T, &fp.c_hi, &fp.c_lo);
    return launch_sampling<In>(fp, stream);
}

}  // namespace osd

using osd::RowStat;

extern "C" osd_status osd_verify_workspace_size(int B, int k, int V, size_t* bytes) {
    if (!bytes || B < 0 || k < 1 || V < 1) return OSD_ERR_INVALID_ARG;
    if (k > OSD_VERIFY_MAX_K || V > OSD_VERIFY_MAX_V) return OSD_ERR_UNSUPPORTED;
    const size_t rows = size_t(B) * size_t(2 * k + 1);
    const size_t need = osd::round256(rows * size_t(osd::verify_slices(B, k, V)) * sizeof(RowStat));
    *bytes = need < 256 ? 256 : need;
    return OSD_OK;
}

extern "C" osd_status osd_verify(const void* draft_logits, const void* target_logits, osd_dtype dtype,
                                 int B, int k, int V, const int32_t* draft_tokens, const float* uniforms,
                                 float temperature, int32_t* accepted, int32_t* out_tokens,
                                 uint8_t* mismatch_mask, float* diag_margin, float* diag_cdf_gap,
                                 void* workspace, size_t workspace_bytes, void* stream) {
    if (dtype != OSD_F32 && dtype != OSD_BF16) return OSD_ERR_INVALID_ARG;
    size_t need = 0;
    const osd_status st = osd_verify_workspace_size(B, k, V, &need);
    if (st != OSD_OK) return st;
    if (!(temperature >= 0.f) || !std::isfinite(temperature)) return OSD_ERR_INVALID_ARG;
    if (B == 0) return OSD_OK;
    const bool greedy = (temperature == 0.f);
    const size_t es = osd::dtype_size(dtype);
    if (!target_logits || !draft_tokens || !accepted || !out_tokens || !mismatch_mask || !workspace)
        return OSD_ERR_INVALID_ARG;
    if (!greedy && (!draft_logits || !uniforms)) return OSD_ERR_INVALID_ARG;
    if (!osd::aligned_to(target_logits, es) || (draft_logits && !osd::aligned_to(draft_logits, es)) ||
        !osd::aligned_to(draft_tokens, 4) || (uniforms && !osd::aligned_to(uniforms, 4)) ||
        !osd::aligned_to(accepted, 4) || !osd::aligned_to(out_tokens, 4) ||
        (diag_margin && !osd::aligned_to(diag_margin, 4)) ||
        (diag_cdf_gap && !osd::aligned_to(diag_cdf_gap, 4)) || !osd::aligned_to(workspace, 16))
        return OSD_ERR_INVALID_ARG;
    if (workspace_bytes < need) return OSD_ERR_INVALID_ARG;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (dtype == OSD_BF16)
        return osd::launch_verify<__nv_bfloat16>(draft_logits, target_logits, B, k, V, draft_tokens, uniforms,
                                                 temperature, accepted, out_tokens, mismatch_mask, diag_margin,
                                                 diag_cdf_gap, static_cast<RowStat*>(workspace), s);
    return osd::launch_verify<float>(draft_logits, target_logits, B, k, V, draft_tokens, uniforms, temperature,
                                     accepted, out_tokens, mismatch_mask, diag_margin, diag_cdf_gap,
                                     static_cast<RowStat*>(workspace), s);
}

// ------------------------------------------------------------------ no-allocation variant
// Some callers cannot call cudaMalloc while they serve: engines that reserve all
// free device memory for their KV cache at start-up and hand out nothing
// afterwards, plugins that run inside such an engine without an allocator of
// their own, and latency-critical loops where cudaMalloc (which may synchronise
// the device) would stall every other stream.  osd_verify_noalloc serves them
// with a fixed workspace that lives in the library itself: a file-scope device
// array, one copy per GPU that loads the library, held until the process exits.
namespace {
constexpr size_t kNoAllocScratchBytes = size_t(4) << 20;  // 4 MiB
constexpr int kNoAllocMaxDevices = 64;
__device__ __align__(256) unsigned char g_verify_scratch[kNoAllocScratchBytes];

// The device address of the array, per device, with the ID of the context it
// was looked up in: a new context (cudaDeviceReset, or a context the caller
// made current) loads the module again, possibly elsewhere, so the address is
// looked up again whenever the current context's ID differs.
struct ScratchSlot {
    unsigned long long ctx_id;
    void* addr;
};
std::mutex g_scratch_mu;
ScratchSlot g_scratch[kNoAllocMaxDevices] = {};

using CtxGetCurrentFn = CUresult (*)(CUcontext*);
using CtxGetIdFn = CUresult (*)(CUcontext, unsigned long long*);

// ID of the context current on the calling thread; false when there is none yet
// (the runtime makes the primary context current on its first device call) or
// the driver does not provide the query.
bool current_context_id(unsigned long long* id) {
    static CtxGetCurrentFn get_current = nullptr;
    static CtxGetIdFn get_id = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void* f = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &f, 12000, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            get_current = reinterpret_cast<CtxGetCurrentFn>(f);
        f = nullptr;
        if (cudaGetDriverEntryPointByVersion("cuCtxGetId", &f, 12000, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            get_id = reinterpret_cast<CtxGetIdFn>(f);
    });
    if (!get_current || !get_id) return false;
    CUcontext ctx = nullptr;
    if (get_current(&ctx) != CUDA_SUCCESS || !ctx) return false;
    return get_id(ctx, id) == CUDA_SUCCESS;
}
}  // namespace

extern "C" osd_status osd_verify_noalloc(const void* draft_logits, const void* target_logits,
                                         osd_dtype dtype, int B, int k, int V,
                                         const int32_t* draft_tokens, const float* uniforms,
                                         float temperature, int32_t* accepted, int32_t* out_tokens,
                                         uint8_t* mismatch_mask, float* diag_margin, float* diag_cdf_gap,
                                         void* stream) {
    size_t need = 0;
    const osd_status st = osd_verify_workspace_size(B, k, V, &need);
    if (st != OSD_OK) return st;
    if (need > kNoAllocScratchBytes) return OSD_ERR_UNSUPPORTED;  // beyond the static scratch
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return OSD_ERR_CUDA;
    if (dev < 0 || dev >= kNoAllocMaxDevices) return OSD_ERR_UNSUPPORTED;
    void* scratch = nullptr;
    {
        // Set-up once per device and context, with that device current: the
        // host-side name of the array is not a device address, so ask the runtime.
        std::lock_guard<std::mutex> lock(g_scratch_mu);
        unsigned long long id = 0;
        const bool have_id = current_context_id(&id);
        ScratchSlot& slot = g_scratch[dev];
        if (!have_id || !slot.addr || slot.ctx_id != id) {
            void* addr = nullptr;
            if (cudaGetSymbolAddress(&addr, g_verify_scratch) != cudaSuccess || !addr) return OSD_ERR_CUDA;
            // the lookup made a context current if none was: key the address on it;
            // without a context ID the address is not cached and is looked up every call
            const bool keyed = have_id || current_context_id(&id);
            slot.addr = keyed ? addr : nullptr;
            slot.ctx_id = keyed ? id : 0ull;
            scratch = addr;
        } else {
            scratch = slot.addr;
        }
    }
    // Only two launches at T = 0 use it: the first writes every entry before the second
    // reads it, so nothing in the shared array needs clearing between calls.
    return osd_verify(draft_logits, target_logits, dtype, B, k, V, draft_tokens, uniforms, temperature,
                      accepted, out_tokens, mismatch_mask, diag_margin, diag_cdf_gap, scratch,
                      kNoAllocScratchBytes, stream);
}
