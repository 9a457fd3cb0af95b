// osd_rowstats.cuh -- row statistics shared by the verifiers (osd_verify.cu,
// osd_tree.cu): at T = 0 a pass with one CTA per (row, vocabulary slice) that
// streams every target row once for the slice's first argmax; at T > 0 the max
// and the sum of 2^((x - max) c) of a cluster CTA's span of a row, taken when the
// row turns out to be needed.
#pragma once

#include <climits>
#include <cstdint>

#include "osd_device.cuh"

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

// One row's statistics from `count` <= 8 partials at x[0], x[stride], ..., merged in
// that order: the maximum first, then the sums brought to it (all loads in flight together).
__device__ __forceinline__ MaxSum merge_slots(const MaxSum* x, int stride, int count, float ch, float cl) {
    MaxSum o[kSeqMaxCluster];
    float m = kNegInf, s = 0.f;
#pragma unroll
    for (int i = 0; i < kSeqMaxCluster; ++i) {
        o[i] = (i < count) ? x[i * stride] : MaxSum{kNegInf, 0.f};
        m = fmaxf(m, o[i].m);
    }
#pragma unroll
    for (int i = 0; i < kSeqMaxCluster; ++i)
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

}  // namespace osd
