// osd_rowstats.cuh -- row statistics shared by the verifiers (osd_verify.cu,
// osd_tree.cu): at T = 0 a pass with one CTA per (row, vocabulary slice) that
// streams every target row once for the slice's first argmax; at T > 0 the max
// and the sum of 2^((x - max) c) of a cluster CTA's span of a row, taken when the
// row turns out to be needed.
#pragma once

#include <climits>
#include <cstdint>

#include "osd_device.cuh"
#include "osd_host.hpp"

namespace osd {

struct RowStat {
    float m;  // max raw logit of the slice
    float s;
    int idx;  // first index of the max
    int pad;
};

constexpr int kStatThreads = 256;
constexpr int kStatUnroll = 2;  // 16-byte vectors per thread per group (one group in flight ahead)

// Vocabulary entries per row_argmax CTA: long slices amortise the per-CTA merge,
// short ones keep enough CTAs in flight when there are few rows.
inline int stats_slice_len(long long rows) {
    return rows >= 2048 ? 32768 : (rows >= 512 ? 16384 : 8192);
}

// ------------------------------------------------------------------ T = 0
template <typename In>
__global__ void __launch_bounds__(kStatThreads)
row_argmax_kernel(const In* __restrict__ target, int V, int slice_len, int n_slices, RowStat* __restrict__ stats) {
    using E = Elem<In>;
    constexpr int kVec = E::kVec;
    __shared__ MaxIdx red_mi[kStatThreads / 32];

    grid_dependency_sync();  // (the consumer of the statistics waits for them in-kernel too)
    const long long item = blockIdx.x;
    const long long row = item / n_slices;
    const int slice = static_cast<int>(item - row * n_slices);
    const int s0 = slice * slice_len;
    const int n = min(V - s0, slice_len);
    const In* p = target + row * V + s0;

    // head (scalar up to the first 16-byte boundary), body (vectors), tail
    const uintptr_t addr = reinterpret_cast<uintptr_t>(p);
    int head = static_cast<int>(((16u - (addr & 15u)) & 15u) / sizeof(In));
    if (head > n) head = n;
    const int nvec = (n - head) / kVec;
    const int tail0 = head + nvec * kVec;
    const In* body = p + head;
    const int tid = threadIdx.x;
    auto load_group = [&](int v, uint4* r) {
#pragma unroll
        for (int u = 0; u < kStatUnroll; ++u) {
            const int vv = v + u * kStatThreads;
            r[u] = (vv < nvec) ? ldg_stream(body + size_t(vv) * kVec) : ninf_raw<In>();
        }
    };
    MaxIdx acc{kNegInf, INT_MAX};
    auto take = [&](float x, int j) {
        if (x > acc.m) { acc.m = x; acc.i = j; }
    };
    if (tid < head) take(E::load(p + tid), s0 + tid);
    uint4 cur[kStatUnroll], nxt[kStatUnroll];
    int v = tid;
    if (v < nvec) load_group(v, cur);
    for (; v < nvec; v += kStatUnroll * kStatThreads) {
        const int vn = v + kStatUnroll * kStatThreads;
        if (vn < nvec) load_group(vn, nxt);
        float cm = E::max_raw(cur[0]);
#pragma unroll
        for (int u = 1; u < kStatUnroll; ++u) cm = fmaxf(cm, E::max_raw(cur[u]));
        if (cm > acc.m) {  // rare: find the first entry equal to the group maximum
#pragma unroll
            for (int u = 0; u < kStatUnroll; ++u) {
                float x[kVec];
                E::unpack(cur[u], x);
                const int j0 = s0 + head + (v + u * kStatThreads) * kVec;
#pragma unroll
                for (int e = 0; e < kVec; ++e) take(x[e], j0 + e);
            }
        }
#pragma unroll
        for (int u = 0; u < kStatUnroll; ++u) cur[u] = nxt[u];
    }
    if (tid < n - tail0) take(E::load(p + tail0 + tid), s0 + tail0 + tid);
    acc = block_reduce<kStatThreads>(acc, [](MaxIdx a, MaxIdx b) { return merge_mi(a, b); }, red_mi);
    if (tid == 0) stats[item] = RowStat{acc.m, 0.f, acc.i, 0};
}

// ------------------------------------------------------------------ rows on demand
// The building blocks of the kernels that give each sequence a thread-block cluster
// and read its rows as they turn out to be needed (osd_verify.cu, osd_tree.cu).
constexpr int kSeqMaxCluster = 8;
constexpr uint64_t kStageWaitNs = 1000000000ull;  // bound on the wait for staged rows ...
constexpr uint64_t kPeerWaitNs = 3000000000ull;   // ... and for the peers' statistics and totals
constexpr size_t kStageMaxSmem = 200 * 1024;      // dynamic shared memory per CTA of the staging kernels
constexpr int kSpanUnroll = 4;  // 16-byte vectors per lane per group (one group in flight ahead)

// Max and sum of 2^((x - max) c) of chunks [c0, c1) of a staged row, by one warp: the
// maximum first, then the sum against it.
template <typename In>
__device__ __forceinline__ MaxSum staged_stats(const In* row, int c0, int c1, float ch, float cl) {
    using E = Elem<In>;
    constexpr int kVec = E::kVec;
    const int lane = threadIdx.x & 31;
    float m = kNegInf;
    for (int c = c0 + lane; c < c1; c += 32) m = fmaxf(m, E::max_raw(lds_v4(row + c * kVec)));
    for (int off = 16; off > 0; off >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, off));
    float2 s2 = f2(0.f);
    if (m != kNegInf) {
        for (int c = c0 + lane; c < c1; c += 32) {
            float2 d[kVec / 2];
            E::minus(lds_v4(row + c * kVec), m, d);
#pragma unroll
            for (int e = 0; e < kVec / 2; ++e) s2 = add2(s2, exp2_pair(d[e], ch, cl));
        }
    }
    float s = s2.x + s2.y;
    for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
    return MaxSum{m, s};
}

// Max and sum of 2^((x - max) c) of the entries p[0, n), taken by `parts` warps:
// this one, number `part`, takes every parts-th group of 32 vectors (part 0 also the
// entries before the first 16-byte boundary, the last part those after the last).
template <typename In>
__device__ __forceinline__ MaxSum span_stats(const In* p, int n, int part, int parts, float c_hi, float c_lo) {
    using E = Elem<In>;
    constexpr int kVec = E::kVec;
    const int lane = threadIdx.x & 31;
    int head = static_cast<int>(((16u - (reinterpret_cast<uintptr_t>(p) & 15u)) & 15u) / sizeof(In));
    if (head > n) head = n;
    const int nvec = (n - head) / kVec;
    const int tail0 = head + nvec * kVec;
    const In* body = p + head;
    float m = kNegInf;
    float2 s2 = f2(0.f);
    auto raise_max = [&](float cm) {
        if (cm > m) {
            s2 = (m == kNegInf) ? f2(0.f) : mul2(s2, f2(ex2(mul_c(m - cm, c_hi, c_lo))));
            m = cm;
        }
    };
    auto one = [&](float x) {
        raise_max(x);
        if (m != kNegInf) s2.x += ex2(mul_c(x - m, c_hi, c_lo));
    };
    const int step = 32 * parts;
    auto load_group = [&](int v, uint4* r) {
#pragma unroll
        for (int u = 0; u < kSpanUnroll; ++u) {
            const int vv = v + u * step;
            r[u] = (vv < nvec) ? ldg_stream(body + size_t(vv) * kVec) : ninf_raw<In>();
        }
    };
    auto absorb = [&](const uint4* r) {
        float cm = E::max_raw(r[0]);
#pragma unroll
        for (int u = 1; u < kSpanUnroll; ++u) cm = fmaxf(cm, E::max_raw(r[u]));
        raise_max(cm);
        if (m != kNegInf) {
#pragma unroll
            for (int u = 0; u < kSpanUnroll; ++u) {
                float2 d[kVec / 2];
                E::minus(r[u], m, d);  // exact, as is c = c_hi + c_lo
#pragma unroll
                for (int e = 0; e < kVec / 2; ++e) s2 = add2(s2, exp2_pair(d[e], c_hi, c_lo));
            }
        }
    };
    // two groups in turn, the next one's loads out before this one's sums
    uint4 ra[kSpanUnroll], rb[kSpanUnroll];
    const int stride = kSpanUnroll * step;
    int v = part * 32 + lane;
    if (v < nvec) load_group(v, ra);
    if (part == 0 && lane < head) one(E::load(p + lane));
    if (part == parts - 1 && lane < n - tail0) one(E::load(p + tail0 + lane));
    for (; v < nvec; v += 2 * stride) {
        if (v + stride < nvec) load_group(v + stride, rb);
        absorb(ra);
        if (v + stride >= nvec) break;
        if (v + 2 * stride < nvec) load_group(v + 2 * stride, ra);
        absorb(rb);
    }
    // warp merge: the maximum first, then one rescale per lane and a plain sum
    float wm = m;
    for (int o = 16; o > 0; o >>= 1) wm = fmaxf(wm, __shfl_xor_sync(0xffffffffu, wm, o));
    float s = (m == kNegInf) ? 0.f : (s2.x + s2.y) * ex2(mul_c(m - wm, c_hi, c_lo));
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    return MaxSum{wm, s};
}

// One row's statistics from `count` <= kMost partials at x[0], x[stride], ..., merged in
// that order: the maximum first, then the sums brought to it (all loads in flight together).
// The caller's bound on its partials is kMost: one that is too low drops part of the row.  (A
// loop over groups of 8 for any count cost the streaming verifier 3 to 6 %, by its spills.)
template <int kMost>
__device__ __forceinline__ MaxSum merge_slots(const MaxSum* x, int stride, int count, float ch, float cl) {
    MaxSum o[kMost];
    float m = kNegInf, s = 0.f;
#pragma unroll
    for (int i = 0; i < kMost; ++i) {
        o[i] = (i < count) ? x[i * stride] : MaxSum{kNegInf, 0.f};
        m = fmaxf(m, o[i].m);
    }
#pragma unroll
    for (int i = 0; i < kMost; ++i)
        if (o[i].m != kNegInf) s += o[i].s * ex2(mul_c(o[i].m - m, ch, cl));
    return MaxSum{m, s};
}

// Four sums over the warp's lanes at once: each exchange halves the number of sums a
// lane carries, 6 shuffles instead of 20, and lane l ends with the total of sum[l / 8].
__device__ __forceinline__ float warp_sum4(const float (&sum)[4]) {
    const int lane = threadIdx.x & 31;
    const bool hi = lane & 16, mid = lane & 8;
    float s01 = hi ? sum[2] : sum[0], s23 = hi ? sum[3] : sum[1];
    s01 += __shfl_xor_sync(0xffffffffu, hi ? sum[0] : sum[2], 16);
    s23 += __shfl_xor_sync(0xffffffffu, hi ? sum[1] : sum[3], 16);
    float tot = mid ? s23 : s01;
    tot += __shfl_xor_sync(0xffffffffu, mid ? s01 : s23, 8);
    for (int o = 4; o > 0; o >>= 1) tot += __shfl_xor_sync(0xffffffffu, tot, o);
    return tot;
}

// ------------------------------------------------------------------ T = 0, rows on demand
// A greedy walk reads a target row only to compare its argmax with the tokens that may
// follow; large batches therefore walk as the samplers do, one cluster per sequence,
// in rounds of a node and the next ones down the walk's likeliest way, four times as
// many after each round.  `Walk` (a kernel parameter) is the chain of a
// draft or a token tree:
//   node_ok(b)          (every thread, strided) whether sequence b's tokens all lie in [0, V)
//   row(b, node)        the node's row among the target rows
//   next(node)          the likeliest child, -1 at a leaf
//   child(b, node, x)   the child whose token is x, -1 if none
//   step(b, depth, child), finish(b, depth, node, x), bad(b): the outputs (one CTA; the
//                       last two by every thread of it)
constexpr int kWalkThreads = 256;
constexpr int kWalkMaxWin = 8;  // nodes per round, a warp or more each

// First argmax of the entries p[0, n) (entry 0 has index j0), shared out as in span_stats.
template <typename In>
__device__ __forceinline__ MaxIdx span_argmax(const In* p, int n, int j0, int part, int parts) {
    using E = Elem<In>;
    constexpr int kVec = E::kVec;
    const int lane = threadIdx.x & 31;
    int head = static_cast<int>(((16u - (reinterpret_cast<uintptr_t>(p) & 15u)) & 15u) / sizeof(In));
    if (head > n) head = n;
    const int nvec = (n - head) / kVec;
    const int tail0 = head + nvec * kVec;
    const In* body = p + head;
    MaxIdx acc{kNegInf, INT_MAX};
    auto take = [&](float x, int j) {
        if (x > acc.m) acc = MaxIdx{x, j};
    };
    const int step = 32 * parts;
    auto load_group = [&](int v, uint4* r) {
#pragma unroll
        for (int u = 0; u < kSpanUnroll; ++u) {
            const int vv = v + u * step;
            r[u] = (vv < nvec) ? ldg_stream(body + size_t(vv) * kVec) : ninf_raw<In>();
        }
    };
    auto absorb = [&](int v, const uint4* r) {
        float cm = E::max_raw(r[0]);
#pragma unroll
        for (int u = 1; u < kSpanUnroll; ++u) cm = fmaxf(cm, E::max_raw(r[u]));
        if (cm > acc.m) {  // rare: find the first entry equal to the group maximum
#pragma unroll
            for (int u = 0; u < kSpanUnroll; ++u) {
                float x[kVec];
                E::unpack(r[u], x);
#pragma unroll
                for (int e = 0; e < kVec; ++e) take(x[e], j0 + head + (v + u * step) * kVec + e);
            }
        }
    };
    if (part == 0 && lane < head) take(E::load(p + lane), j0 + lane);
    uint4 ra[kSpanUnroll], rb[kSpanUnroll];
    const int stride = kSpanUnroll * step;
    int v = part * 32 + lane;
    if (v < nvec) load_group(v, ra);
    for (; v < nvec; v += 2 * stride) {
        if (v + stride < nvec) load_group(v + stride, rb);
        absorb(v, ra);
        if (v + stride >= nvec) break;
        if (v + 2 * stride < nvec) load_group(v + 2 * stride, ra);
        absorb(v + stride, rb);
    }
    if (part == parts - 1 && lane < n - tail0) take(E::load(p + tail0 + lane), j0 + tail0 + lane);
    return warp_reduce(acc, [](MaxIdx a, MaxIdx b) { return merge_mi(a, b); });
}

template <typename In, typename Walk>
__global__ void __launch_bounds__(kWalkThreads, 4)
greedy_walk_kernel(Walk wk, const In* target, int V, int csize, int span, int win) {
    constexpr int kWarps = kWalkThreads / 32;
    __shared__ MaxIdx s_part[kWarps];
    __shared__ __align__(8) MaxIdx s_recv[2][kSeqMaxCluster * kWalkMaxWin];  // [CTA][node], two rounds
    __shared__ __align__(8) uint64_t s_bar[2];
    __shared__ int s_best[kWalkMaxWin];
    __shared__ int s_node, s_depth, s_state;  // state: 0 another round, 1 done, 2 a wait gave up
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int rank = (csize > 1) ? static_cast<int>(cluster_rank()) : 0;
    const int b = blockIdx.x / csize;
    const int e0 = rank * span, n = min(span, V - e0);
    if (tid == 0) {
        mbar_init_only(&s_bar[0], 1);
        mbar_init_only(&s_bar[1], 1);
        fence_mbarrier_init();
        s_node = 0;
        s_depth = 0;
    }
    grid_dependency_sync();
    const int bad = wk.node_ok(b) ? 0 : 1;
    if (__syncthreads_or(bad)) {  // uniform over the cluster, before any push to a peer
        if (rank == 0) wk.bad(b);
        return;
    }
    // the barriers are initialised before any peer pushes to them: arrive now, wait before the first push
    if (csize > 1) cluster_arrive_relaxed();
    for (unsigned round = 0;; ++round) {
        const int node = s_node;
        int w = 1;
        for (int nd = wk.next(node); nd >= 0 && w < win; nd = wk.next(nd)) ++w;
        const int parts = kWarps / w;
        const int q = warp / parts;
        if (q < w) {
            int nd = node;
            for (int i = 0; i < q; ++i) nd = wk.next(nd);
            const MaxIdx mine = span_argmax<In>(target + wk.row(b, nd) * V + e0, n, e0, warp - q * parts, parts);
            if (lane == 0) s_part[warp] = mine;
        }
        __syncthreads();
        if (round == 0 && csize > 1) asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
        if (warp == 0) {
            const unsigned buf = round & 1u;
            MaxIdx* recv = s_recv[buf];
            bool gone = false;
            MaxIdx acc{kNegInf, INT_MAX};
            if (lane < w) {
                for (int x = 0; x < parts; ++x) acc = merge_mi(acc, s_part[lane * parts + x]);
                for (int c = 0; c < csize && csize > 1; ++c)
                    st_async_v2(map_rank(&recv[rank * kWalkMaxWin + lane], static_cast<uint32_t>(c)),
                                make_float2(acc.m, __int_as_float(acc.i)), map_rank(&s_bar[buf], static_cast<uint32_t>(c)));
            }
            if (csize > 1) {
                if (lane == 0) mbar_arrive_expect_tx(&s_bar[buf], static_cast<uint32_t>(csize * w) * 8u);
                gone = !mbar_wait_cluster_bounded(&s_bar[buf], (round >> 1) & 1u, kPeerWaitNs);
                acc = MaxIdx{kNegInf, INT_MAX};
                if (!gone && lane < w)
                    for (int c = 0; c < csize; ++c) acc = merge_mi(acc, recv[c * kWalkMaxWin + lane]);
            }
            if (lane < w) s_best[lane] = acc.i == INT_MAX ? 0 : acc.i;
            gone = __any_sync(0xffffffffu, gone);
            __syncwarp();
            if (lane == 0) {
                int nd = node, depth = s_depth, state = gone ? 2 : 1;
                for (int i = 0; i < w && state == 1; ++i) {
                    const int ch = wk.child(b, nd, s_best[i]);
                    if (ch < 0) {
                        s_best[0] = s_best[i];  // the walk ends at nd, with its argmax as the extra token
                        break;
                    }
                    if (rank == 0) wk.step(b, depth, ch);
                    ++depth;
                    if (i + 1 == w || ch != wk.next(nd)) state = 0;
                    nd = ch;
                }
                s_node = nd;
                s_depth = depth;
                s_state = state;
            }
        }
        __syncthreads();
        if (s_state) {
            if (s_state == 2 && csize > 1 && tid == 0)
                mbar_wait_cluster_bounded(&s_bar[round & 1u], (round >> 1) & 1u, kPeerWaitNs);
            break;
        }
        win = min(4 * win, kWalkMaxWin);
    }
    if (rank != 0) return;
    if (s_state == 2) wk.bad(b);  // the peers' argmaxes did not arrive in time: reported as bad
    else wk.finish(b, s_depth, s_node, s_best[0]);
}

// Launch a greedy walk over B sequences of `rows` rows each, at most `depth` of them on any
// walk, or return false where the pass over every row does better: that one reads at the copy
// bandwidth, a walk pays about 2.5 us a round.  Trees, of which a walk sees the smaller part,
// from 20 MB and 8 sequences on (27 nodes: 16 x 32000 8.7 -> 5.1 us, 64 x 100000 58 -> 15,
// 48 x 128256 fp32 96 -> 20; 2 x 135808 fp32 8.9 against 9.3); chains only where one position is
// 40 MB (256 x 9 x 128256: 90 us, on demand 27 with 0.02 accepted, 54 with 0.9, 77 with 3.5 and
// 100 with 6.4; 32 x 9 x 128256, 8 MB: 16.4 against 6.9 and 21 with the first and the last draft).
template <typename In, typename Walk>
static bool launch_greedy_walk(const Walk& wk, const In* target, int B, int rows, int depth, int V, cudaStream_t stream,
                               osd_status* st) {
    const double pos = double(B) * V * double(sizeof(In));  // bytes of one node of the batch
    if (pos < 40e6 && (B < 8 || rows < 2 * depth || pos * rows < 20e6)) return false;
    const int win = pos <= 4e6 ? 4 : (pos <= 16e6 ? 2 : 1);
    int c = kSeqMaxCluster;
    while (c > 1 && (V <= 2048 * c || ((long long)B * c / 2 >= 3LL * device_sms() && size_t(V / (c / 2)) * sizeof(In) <= 68 * 1024)))
        c /= 2;
    const int span = ((V + c - 1) / c + 63) / 64 * 64;
    const int csize = (V + span - 1) / span;
    if ((long long)B * csize > INT_MAX) return false;
    *st = from_cuda(launch_ex(true, greedy_walk_kernel<In, Walk>, dim3(unsigned(B) * unsigned(csize)), dim3(kWalkThreads), 0,
                              stream, csize, wk, target, V, csize, span, win));
    return true;
}

}  // namespace osd
