// osd_tree.cu -- multi-candidate verification over a token tree (the tree-style
// speculative decoding the paper runs OSD on with Medusa heads: several
// candidates per position) on sm_103a.
//
// T > 0: one launch, tree_walk_kernel, one thread-block cluster per sequence, which
// walks the tree from the root.  At a node it tests the children in index order
// with the accept rule of Appendix A.1 against the current residual.  After j
// rejections the residual is norm(max(0, p - s_j q)) with s_0 = 0 and
// s_{j+1} = s_j + N_j, N_j = sum max(0, p - s_j q), so child y passes iff
// u < max(0, p(y)/q(y) - s_j) / N_j.  Every rejection costs one cluster-wide pass
// that recomputes N_{j+1}; an acceptance moves the walk to the child.  When no child
// passes, the extra token is drawn from max(0, p - s q) by inverse CDF from the
// sub-tile sums of the last pass, as the verifier draws its residual token (masses
// summed in exact 64-bit fixed point).  Only the rows the walk comes to are read.
//
// T = 0: greedy_walk_kernel (osd_rowstats.cuh), which reads the target rows of the
// matching children on its way; where the tree is small or little more than a
// chain, two launches, row_argmax_kernel over every target row's slices and
// tree_greedy_kernel, which follows the matching children.
#include <algorithm>
#include <climits>
#include <cmath>
#include <cstdint>

#include "osd.h"
#include "osd_device.cuh"
#include "osd_host.hpp"
#include "osd_rowstats.cuh"

namespace osd {

constexpr int kTreeThreads = 256;
constexpr int kTreeWarps = kTreeThreads / 32;
constexpr int kTreeMaxWin = 4;                  // nodes per round ...
constexpr int kTreeMaxRows = 2 * kTreeMaxWin;   // ... and their rows
constexpr int kTreeUnroll = 4;                  // sub-tiles of loads in flight per warp in a mass pass
constexpr int kGreedyThreads = 128;

// Children lists of the static tree: first child and next sibling, increasing
// index; and each node's parent (-1 at the root).
struct TreeTopo {
    int8_t first_child[OSD_TREE_MAX_NODES];
    int8_t next_sibling[OSD_TREE_MAX_NODES];
    int8_t parent[OSD_TREE_MAX_NODES];
};

struct TreeParams {
    const void* draft;
    const void* target;
    int n, V;  // nodes per tree, vocabulary
    const int32_t* tokens;
    const float* uniforms;
    float T, c_hi, c_lo;
    const RowStat* stats;  // T = 0: the target rows' slice argmaxes
    int n_slices;
    int32_t* accepted;
    int32_t* path;
    int32_t* out_tokens;
    int32_t* last_node;
    float* diag_margin;
    float* diag_gap;
    int csize, span;
    TreeTopo topo;
};

// T = 0: the walk follows the child whose token is the target argmax.  One CTA per sequence.
__global__ void __launch_bounds__(kGreedyThreads) tree_greedy_kernel(TreeParams p) {
    __shared__ int s_nidx[OSD_TREE_MAX_NODES];
    const int tid = threadIdx.x, b = blockIdx.x, n = p.n;
    const int32_t* y = p.tokens + size_t(b) * n;
    int32_t* pth = p.path + size_t(b) * n;
    int32_t* out = p.out_tokens + size_t(b) * n;
    int bad = 0;
    for (int i = 1 + tid; i < n; i += kGreedyThreads) bad |= (y[i] < 0 || y[i] >= p.V) ? 1 : 0;
    bad = __syncthreads_or(bad);
    for (int i = tid; i < n; i += kGreedyThreads) {
        pth[i] = -1;
        out[i] = -1;
        if (p.diag_margin) p.diag_margin[size_t(b) * n + i] = __int_as_float(0x7fc00000);
    }
    if (tid == 0) {
        if (p.diag_gap) p.diag_gap[b] = __int_as_float(0x7fc00000);
        if (bad) {
            p.accepted[b] = -1;
            p.last_node[b] = -1;
        }
    }
    // the row statistics are complete from here on.  A bad sequence waits for them too: the grid
    // must not end before row_argmax_kernel has, since the next call on the stream waits for this
    // grid alone before it writes the workspace again (or the logits, which that kernel reads).
    grid_dependency_sync();
    if (bad) return;
    for (int nd = tid; nd < n; nd += kGreedyThreads) {
        const RowStat* st = p.stats + (size_t(b) * n + nd) * p.n_slices;
        MaxIdx acc{kNegInf, INT_MAX};
#pragma unroll 4
        for (int sl = 0; sl < p.n_slices; ++sl) acc = merge_mi(acc, MaxIdx{st[sl].m, st[sl].idx});
        s_nidx[nd] = (acc.i == INT_MAX) ? 0 : acc.i;
    }
    __syncthreads();  // (the initialisation above lands before the walk writes its entries)
    if (tid != 0) return;
    int node = 0, depth = 0;
    for (;;) {
        const int best = s_nidx[node];
        int next = -1;
        for (int c = p.topo.first_child[node]; c >= 0; c = p.topo.next_sibling[c])
            if (y[c] == best) { next = c; break; }
        if (next < 0) {
            out[depth] = best;
            break;
        }
        pth[depth] = next;
        out[depth++] = y[next];
        node = next;
    }
    p.accepted[b] = depth;
    p.last_node[b] = node;
}

// The same walk on demand (osd_rowstats.cuh).
struct GreedyTree {
    TreeParams p;
    __device__ bool node_ok(int b) const {
        bool ok = true;
        for (int i = 1 + threadIdx.x; i < p.n; i += kWalkThreads) {
            const int y = p.tokens[size_t(b) * p.n + i];
            ok = ok && y >= 0 && y < p.V;
        }
        return ok;
    }
    __device__ size_t row(int b, int nd) const { return size_t(b) * p.n + nd; }
    __device__ int next(int nd) const { return p.topo.first_child[nd]; }
    __device__ int child(int b, int nd, int x) const {
        for (int c = p.topo.first_child[nd]; c >= 0; c = p.topo.next_sibling[c])
            if (p.tokens[size_t(b) * p.n + c] == x) return c;
        return -1;
    }
    __device__ void step(int b, int depth, int c) const {
        p.path[size_t(b) * p.n + depth] = c;
        p.out_tokens[size_t(b) * p.n + depth] = p.tokens[size_t(b) * p.n + c];
    }
    __device__ void finish(int b, int depth, int nd, int x) const {
        for (int i = threadIdx.x; i < p.n; i += kWalkThreads) {
            if (i >= depth) p.path[size_t(b) * p.n + i] = -1;
            if (i >= depth) p.out_tokens[size_t(b) * p.n + i] = i == depth ? x : -1;
            if (p.diag_margin) p.diag_margin[size_t(b) * p.n + i] = __int_as_float(0x7fc00000);
        }
        if (threadIdx.x == 0) {
            p.accepted[b] = depth;
            p.last_node[b] = nd;
            if (p.diag_gap) p.diag_gap[b] = __int_as_float(0x7fc00000);
        }
    }
    __device__ void bad(int b) const {
        finish(b, 0, -1, -1);
        if (threadIdx.x == 0) p.accepted[b] = -1;
    }
};

// T > 0.  Each CTA owns a span of the vocabulary.  A round takes the rows of a node and of
// the `win` - 1 next ones down its first children (the likeliest way on).  The span
// statistics meet by st.async, every CTA merging the same slots in rank order, and
// warp 0 of every CTA walks on alike: tests cost no exchange until a rejection needs
// a mass pass, whose span totals meet the same way, or the walk leaves the round.
//
// What bounds it: the chain of dependent phases, about 3 us a round and 2 us a rejection.
// B = 32, 27 nodes, V = 32000 (1.8 accepted): 23.3 us where the statistics of every node's rows
// took 43.8; V = 128256: 48 us against 125; B = 64, V = 32001: 41 us against 109.  Two CTAs an SM
// at 120 registers: with three or four the passes spill (33 and 35 us, where two took 24); rows
// staged in shared memory first took 26 us, and at V = 128256, where they leave one CTA an SM, 79 us.
template <typename In, bool kAligned>
__global__ void __launch_bounds__(kTreeThreads) tree_walk_kernel(TreeParams p, int win) {
    using E = Elem<In>;
    constexpr int kW = E::kVec;  // entries per lane per sub-tile
    constexpr int kSub = 32 * kW;
    extern __shared__ float s_sub[];  // mass of every sub-tile of this CTA's span (last pass)
    __shared__ MaxSum s_part[kTreeMaxRows > kTreeWarps ? kTreeMaxRows : kTreeWarps];
    __shared__ __align__(8) MaxSum s_recv[2][kSeqMaxCluster * kTreeMaxRows];  // [CTA][row slot], two rounds
    __shared__ __align__(8) unsigned long long s_totals[2][kSeqMaxCluster];   // span masses, two passes
    __shared__ __align__(8) uint64_t s_bar[2], s_tbar[2];
    // the round's statistics: row slot 2 q is node q's target row, 2 q + 1 its draft row
    __shared__ float s_m[kTreeMaxRows], s_s[kTreeMaxRows];
    __shared__ double s_ratio[kTreeMaxWin];  // E_z / E_t of each node with children
    // per child c: its token's logits in the draft and target rows of its parent, and its uniform
    __shared__ float s_zy[OSD_TREE_MAX_NODES], s_ty[OSD_TREE_MAX_NODES], s_u[OSD_TREE_MAX_NODES];
    __shared__ int s_y[OSD_TREE_MAX_NODES];
    __shared__ int s_act, s_node, s_q, s_depth;  // what warp 0 decided
    __shared__ float s_shift;

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int csize = p.csize;
    const int rank = (csize > 1) ? static_cast<int>(cluster_rank()) : 0;
    const int b = blockIdx.x / csize;
    const int n = p.n, V = p.V;
    const int e0 = rank * p.span;
    const int cnt = min(p.span, V - e0);
    const int nsub = (cnt + kSub - 1) / kSub;
    const In* draft = static_cast<const In*>(p.draft) + size_t(b) * n * V;
    const In* target = static_cast<const In*>(p.target) + size_t(b) * n * V;
    int32_t* pth = p.path + size_t(b) * n;
    int32_t* out = p.out_tokens + size_t(b) * n;
    const float ch = p.c_hi, cl = p.c_lo;

    // nodes of the round that starts at `node`: down the first children; and their rows
    // (a leaf, which only the last can be, has no use for its draft row)
    auto round_nodes = [&](int node) {
        int w = 1;
        for (int nd = p.topo.first_child[node]; nd >= 0 && w < win; nd = p.topo.first_child[nd]) ++w;
        return w;
    };
    auto node_at = [&](int node, int q) {
        for (; q > 0; --q) node = p.topo.first_child[node];
        return node;
    };
    auto row_of = [&](int node, int slot) {
        const size_t nd = static_cast<size_t>(node_at(node, slot >> 1));
        return ((slot & 1) ? draft : target) + nd * V + e0;
    };
    auto rows_of = [&](int node, int w) { return 2 * w - (p.topo.first_child[node_at(node, w - 1)] < 0 ? 1 : 0); };

    if (tid == 0) {
        for (int i = 0; i < 2; ++i) {
            mbar_init_only(&s_bar[i], 1);
            mbar_init_only(&s_tbar[i], 1);
        }
        fence_mbarrier_init();
    }
    grid_dependency_sync();
    // check the tokens and gather the two logits every child's accept test needs
    int bad = 0;
    for (int i = tid; i < n; i += kTreeThreads) {
        s_u[i] = p.uniforms[size_t(b) * n + i];
        const int yi = p.tokens[size_t(b) * n + i];
        s_y[i] = yi;
        if (i == 0) continue;
        if (yi < 0 || yi >= V) {
            bad = 1;
        } else {
            const size_t prow = static_cast<size_t>(p.topo.parent[i]) * V;
            s_zy[i] = E::load(draft + prow + yi);
            s_ty[i] = E::load(target + prow + yi);
        }
    }
    if (rank == 0 && p.diag_margin)
        for (int i = tid; i < n; i += kTreeThreads) p.diag_margin[size_t(b) * n + i] = __int_as_float(0x7fc00000);
    __syncthreads();  // the barriers are initialised before anyone waits on them
    // ... and before any peer pushes to them: arrive now, wait before the first push
    if (csize > 1) cluster_arrive_relaxed();

    constexpr int kRound = 0, kMass = 1, kDraw = 2, kGone = 3, kBad = 4;  // what comes next
    int act = kRound, node = 0;  // node: the round's first
    unsigned round = 0, pass = 0;

    // warp 0's walk state (the same in every CTA): the current node, its place in the
    // round, the child under test, the residual's shift and mass
    int cur = 0, q = 0, child = p.topo.first_child[0], depth = 0;
    float s = 0.f;
    double N = 1.0;
    unsigned long long Nfix = 0ull;
    int rn_nodes = 1;
    // Test children from `child` on until something else has to happen; every lane alike.
    auto walk = [&]() {
        for (;;) {
            if (child < 0) {  // no child passed: draw, from p itself when none was rejected
                act = (s > 0.f) ? kDraw : kMass;
                return;
            }
            // p(y)/q(y) from the logit differences and the two sums, as the verifier
            // forms it; the test u < max(0, p/q - s) / N is taken as u N < max(0, p/q - s)
            const float zt = s_zy[child], tt = s_ty[child];
            double rn;  // max(0, p(y)/q(y) - s_j)
            if (zt == kNegInf) {
                rn = (tt > kNegInf) ? INFINITY : 0.0;
            } else {
                const float D = (tt - s_m[2 * q]) - (zt - s_m[2 * q + 1]);
                const double rho = double(ex2(mul_c(D, ch, cl))) * s_ratio[q];
                rn = fmax(rho - double(s), 0.0);
            }
            const float uc = s_u[child];
            if (rank == 0 && lane == 0 && p.diag_margin)  // |u - r|, a diagnostic: fp32 is enough
                p.diag_margin[size_t(b) * n + child] = fabsf(uc - float(rn) / float(N));
            if (!(double(uc) * N < rn)) {
                s = static_cast<float>(double(s) + N);  // rejected: s_{j+1} = s_j + N_j
                act = kMass;
                return;
            }
            if (rank == 0 && lane == 0) {
                pth[depth] = child;
                out[depth] = s_y[child];
            }
            ++depth;
            const bool next_in_round = q + 1 < rn_nodes && child == p.topo.first_child[cur];
            cur = child;
            child = p.topo.first_child[cur];
            s = 0.f;
            N = 1.0;
            if (!next_in_round) {
                act = kRound;
                return;
            }
            ++q;
        }
    };
    auto publish = [&]() {
        if (lane == 0) {
            s_act = act;
            s_node = cur;
            s_q = q;
            s_shift = s;
            s_depth = depth;
        }
    };
    struct Raw {
        uint4 t, z;
    };
    auto load_sub = [&](const In* trow, const In* zrow, bool use_q, int sb, Raw& r) {
        const int j0 = sb * kSub + lane * kW;  // in the span
        const int m = min(kW, cnt - j0);
        bool whole = m == kW;
        if constexpr (!kAligned)
            whole = whole && shifted_inside(trow - e0, e0 + j0, V) && (!use_q || shifted_inside(zrow - e0, e0 + j0, V));
        if (whole) {
            if constexpr (kAligned) {
                r.t = ldg_stream(trow + j0);
                r.z = use_q ? ldg_stream(zrow + j0) : r.t;
            } else {
                r.t = ldg_shifted(trow + j0);
                r.z = use_q ? ldg_shifted(zrow + j0) : r.t;
            }
        } else {
            float tv[kW], zv[kW];
#pragma unroll
            for (int e = 0; e < kW; ++e) {
                tv[e] = (e < m) ? E::load(trow + j0 + e) : kNegInf;
                zv[e] = (e < m && use_q) ? E::load(zrow + j0 + e) : kNegInf;
            }
            r.t = pack_raw<In, kW>(tv);
            r.z = pack_raw<In, kW>(zv);
        }
    };
    // w = max(0, p - s q) of kW entries of one lane (p itself when !use_q), in pairs
    auto weights = [&](const Raw& r, bool use_q, float sh, float mt, float inv_st, float mz, float inv_sz, float2* w) {
        float2 d[kW / 2];
        E::minus(r.t, mt, d);
#pragma unroll
        for (int e = 0; e < kW / 2; ++e) w[e] = mul2(exp2_pair(d[e], ch, cl), f2(inv_st));
        if (use_q) {
            E::minus(r.z, mz, d);
#pragma unroll
            for (int e = 0; e < kW / 2; ++e) {
                const float2 qj = mul2(exp2_pair(d[e], ch, cl), f2(inv_sz));
                const float2 df = fma2(f2(-sh), qj, w[e]);
                w[e] = make_float2(fmaxf(df.x, 0.f), fmaxf(df.y, 0.f));
            }
        }
    };

    for (;;) {
        if (act == kRound) {
            // ---- the round's rows: span statistics, exchanged and merged
            const int w = round_nodes(node), nr = rows_of(node, w);
            const int parts = max(1, kTreeWarps / nr);
            for (int it = warp; it < nr * parts; it += kTreeWarps) {
                const int r = it / parts;
                const MaxSum mine = span_stats<In>(row_of(node, r), cnt, it - r * parts, parts, ch, cl);
                if (lane == 0) s_part[it] = mine;
            }
            if (__syncthreads_or(bad)) {  // (only in the first round) uniform over the cluster, before any push to a peer
                act = kBad;
                break;
            }
            if (round == 0 && csize > 1) asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
            if (warp == 0) {
                const unsigned buf = round & 1u;
                MaxSum* recv = s_recv[buf];
                bool gone = false;
                if (lane < nr) {
                    const MaxSum acc = merge_slots<kTreeWarps>(s_part + lane * parts, 1, parts, ch, cl);
                    if (csize > 1) {
                        for (int d = 0; d < csize; ++d)
                            st_async_v2(map_rank(&recv[rank * kTreeMaxRows + lane], static_cast<uint32_t>(d)),
                                        make_float2(acc.m, acc.s), map_rank(&s_bar[buf], static_cast<uint32_t>(d)));
                    } else {
                        recv[lane] = acc;
                    }
                }
                if (csize > 1) {
                    if (lane == 0) mbar_arrive_expect_tx(&s_bar[buf], static_cast<uint32_t>(csize * nr) * 8u);
                    gone = !mbar_wait_cluster_bounded(&s_bar[buf], (round >> 1) & 1u, kPeerWaitNs);
                }
                __syncwarp();
                if (!gone && lane < nr) {
                    const MaxSum o = merge_slots<kSeqMaxCluster>(recv + lane, kTreeMaxRows, csize, ch, cl);
                    s_m[lane] = o.m;
                    s_s[lane] = o.s;
                }
                __syncwarp();
                if (2 * lane + 1 < nr) s_ratio[lane] = double(s_s[2 * lane + 1]) / double(s_s[2 * lane]);
                __syncwarp();
                q = 0;
                rn_nodes = w;
                if (__any_sync(0xffffffffu, gone)) act = kGone;
                else walk();
                publish();
            }
            ++round;
        } else {
            // ---- one cluster-wide pass: the mass of every sub-tile of w = max(0, p - s q) (of p
            // itself at a node without a rejection, to draw from) into s_sub, and the row's mass
            const int nq = s_q;
            const float sh = s_shift;
            const bool use_q = sh > 0.f;
            const int nd = s_node;
            const In* trow = target + size_t(nd) * V + e0;
            const In* zrow = draft + size_t(nd) * V + e0;
            const float mt = s_m[2 * nq], inv_st = 1.0f / s_s[2 * nq];
            const float mz = use_q ? s_m[2 * nq + 1] : 0.f, inv_sz = use_q ? 1.0f / s_s[2 * nq + 1] : 0.f;
            for (int sb0 = warp; sb0 < nsub; sb0 += kTreeWarps * kTreeUnroll) {
                Raw r[kTreeUnroll];  // the loads of kTreeUnroll sub-tiles go out together
#pragma unroll
                for (int u2 = 0; u2 < kTreeUnroll; ++u2)
                    if (sb0 + u2 * kTreeWarps < nsub) load_sub(trow, zrow, use_q, sb0 + u2 * kTreeWarps, r[u2]);
                float sum[kTreeUnroll];
#pragma unroll
                for (int u2 = 0; u2 < kTreeUnroll; ++u2) {
                    sum[u2] = 0.f;
                    if (sb0 + u2 * kTreeWarps < nsub) {
                        float2 wv[kW / 2];
                        weights(r[u2], use_q, sh, mt, inv_st, mz, inv_sz, wv);
                        float2 s2 = wv[0];
#pragma unroll
                        for (int e = 1; e < kW / 2; ++e) s2 = add2(s2, wv[e]);
                        sum[u2] = s2.x + s2.y;
                    }
                }
                const float tot = warp_sum4(sum);
                const int sb = sb0 + (lane >> 3) * kTreeWarps;
                if ((lane & 7) == 0 && sb < nsub) s_sub[sb] = tot;
            }
            __syncthreads();
            if (warp == 0) {
                unsigned long long part = 0ull;
                for (int sb = lane; sb < nsub; sb += 32) part += fix_of(s_sub[sb]);
                part = warp_sum_u64(part);
                const unsigned buf = pass & 1u;
                bool gone = false;
                if (csize > 1) {
                    if (lane < csize)
                        st_async_u64(map_rank(&s_totals[buf][rank], static_cast<uint32_t>(lane)), part,
                                     map_rank(&s_tbar[buf], static_cast<uint32_t>(lane)));
                    if (lane == 0) mbar_arrive_expect_tx(&s_tbar[buf], static_cast<uint32_t>(csize) * 8u);
                    gone = !mbar_wait_cluster_bounded(&s_tbar[buf], (pass >> 1) & 1u, kPeerWaitNs);
                }
                const unsigned long long tot = lane < csize ? (csize > 1 ? s_totals[buf][lane] : part) : 0ull;
                Nfix = __shfl_sync(0xffffffffu, warp_incl_scan_u64(tot), 31);
                if (__any_sync(0xffffffffu, gone)) {
                    act = kGone;
                } else if (!use_q) {  // a leaf, or a node whose draw is from p itself
                    act = kDraw;
                } else {
                    N = __ull2double_rn(Nfix) * (1.0 / static_cast<double>(1ull << kFixBits));
                    child = p.topo.next_sibling[child];
                    walk();
                }
                publish();
            }
            ++pass;
        }
        __syncthreads();
        act = s_act;
        node = s_node;
        if (act == kDraw || act == kGone) break;
    }
    if (act != kDraw) {  // a bad token, or the GPU did not deliver in time: the sequence is reported as bad
        if (act == kGone && csize > 1 && tid == 0) {
            if (round > 0) mbar_wait_cluster_bounded(&s_bar[(round - 1) & 1u], ((round - 1) >> 1) & 1u, kPeerWaitNs);
            if (pass > 0) mbar_wait_cluster_bounded(&s_tbar[(pass - 1) & 1u], ((pass - 1) >> 1) & 1u, kPeerWaitNs);
        }
        if (rank == 0) {
            for (int i = tid; i < n; i += kTreeThreads) {
                pth[i] = -1;
                out[i] = -1;
                if (p.diag_margin) p.diag_margin[size_t(b) * n + i] = __int_as_float(0x7fc00000);
            }
            if (tid == 0) {
                p.accepted[b] = -1;
                p.last_node[b] = -1;
                if (p.diag_gap) p.diag_gap[b] = __int_as_float(0x7fc00000);
            }
        }
        return;
    }
    // ---- the walk's outputs, and the extra token (entry `depth`) by the CTA that owns it
    depth = s_depth;
    if (rank == 0) {
        if (tid == 0) {
            p.accepted[b] = depth;
            p.last_node[b] = node;
        }
        for (int i = tid; i < n; i += kTreeThreads) {
            if (i >= depth) pth[i] = -1;
            if (i > depth) out[i] = -1;
        }
    }
    if (warp != 0) return;
    // the last pass's span masses, a lane per CTA: W, tau = floor(u W) and the owning CTA
    const unsigned lastbuf = (pass - 1) & 1u;
    unsigned long long own = 0ull;
    if (csize == 1) {
        for (int sb = lane; sb < nsub; sb += 32) own += fix_of(s_sub[sb]);
        own = warp_sum_u64(own);
    }
    const unsigned long long tot = lane < csize ? (csize > 1 ? s_totals[lastbuf][lane] : own) : 0ull;
    const unsigned long long incl = warp_incl_scan_u64(tot);
    const unsigned long long W = __shfl_sync(0xffffffffu, incl, 31);
    const unsigned long long tau = fix_scale(s_u[0], W);
    int owner = 0, mode = 0;  // mode 0: inverse CDF, 1: largest positive entry, 2: argmax p
    unsigned long long base = 0ull;
    if (W > 0ull) {
        const unsigned hit = __ballot_sync(0xffffffffu, lane < csize && incl > tau);
        if (hit) {
            owner = __ffs(hit) - 1;
            base = __shfl_sync(0xffffffffu, incl - tot, owner);
        } else {
            mode = 1;
            owner = 31 - __clz(__ballot_sync(0xffffffffu, lane < csize && tot > 0ull));
        }
    } else {
        mode = 2;
    }
    if (rank != owner) return;
    const int nq = s_q;
    const float sh = s_shift;
    const bool use_q = sh > 0.f;
    const In* trow = target + size_t(node) * V + e0;
    const In* zrow = draft + size_t(node) * V + e0;
    int pick = -1;
    float gap = __int_as_float(0x7fc00000);
    if (mode == 2) {  // no residual mass: argmax of p over the row, lowest index
        const In* grow = target + size_t(node) * V;
        MaxIdx acc{kNegInf, INT_MAX};
        for (int j = lane; j < V; j += 32) {
            const float t = E::load(grow + j);
            if (t > acc.m) { acc.m = t; acc.i = j; }
        }
        acc = warp_reduce(acc, [](MaxIdx x, MaxIdx z) { return merge_mi(x, z); });
        if (lane == 0) pick = (acc.i == INT_MAX) ? 0 : acc.i;
    } else {
        // the sub-tile: lane l owns the run [s_lo, s_hi) of sub-tiles
        const int per = (nsub + 31) / 32;
        const int s_lo = min(nsub, lane * per), s_hi = min(nsub, s_lo + per);
        unsigned long long mine = 0ull;
        for (int sb = s_lo; sb < s_hi; ++sb) mine += fix_of(s_sub[sb]);
        const unsigned long long excl = base + warp_incl_scan_u64(mine) - mine;
        int tile = -1;
        unsigned long long tbase = 0ull;
        if (mode == 0) {
            const unsigned h = __ballot_sync(0xffffffffu, excl <= tau && excl + mine > tau);
            if (h) {
                const int l = __ffs(h) - 1;
                if (lane == l) {  // the sums are exact: the run holds tau in one sub-tile
                    unsigned long long c2 = excl;
                    for (int sb = s_lo; sb < s_hi; ++sb) {
                        const unsigned long long v = fix_of(s_sub[sb]);
                        if (c2 + v > tau) { tile = sb; break; }
                        c2 += v;
                    }
                    tbase = c2;
                }
                tile = __shfl_sync(0xffffffffu, tile, l);
                tbase = __shfl_sync(0xffffffffu, tbase, l);
            } else {
                mode = 1;
            }
        }
        if (mode == 1) {
            int last = -1;
            for (int sb = s_lo; sb < s_hi; ++sb)
                if (s_sub[sb] > 0.f) last = sb;
            for (int o = 16; o > 0; o >>= 1) last = max(last, __shfl_xor_sync(0xffffffffu, last, o));
            tile = max(last, 0);
        }
        Raw r;
        load_sub(trow, zrow, use_q, tile, r);
        float2 w2[kW / 2];
        weights(r, use_q, sh, s_m[2 * nq], 1.0f / s_s[2 * nq], use_q ? s_m[2 * nq + 1] : 0.f,
                use_q ? 1.0f / s_s[2 * nq + 1] : 0.f, w2);
        float wv[kW];
#pragma unroll
        for (int e = 0; e < kW / 2; ++e) {
            wv[2 * e] = w2[e].x;
            wv[2 * e + 1] = w2[e].y;
        }
        const int j0 = e0 + tile * kSub + lane * kW;
        bool done = false;
        if (mode == 0) {
            unsigned long long wsum = 0ull;
#pragma unroll
            for (int e = 0; e < kW; ++e) wsum += fix_of(wv[e]);
            const unsigned long long wex = tbase + warp_incl_scan_u64(wsum) - wsum;
            const bool hit = wex <= tau && wex + wsum > tau;
            if (hit) {
                unsigned long long C = wex;
                for (int e = 0; e < kW; ++e) {
                    const unsigned long long Cprev = C;
                    C += fix_of(wv[e]);
                    if (C > tau) {
                        pick = j0 + e;
                        gap = fminf(fix_to_float(C - tau), fix_to_float(tau - Cprev)) / fix_to_float(W);
                        break;
                    }
                }
            }
            done = __any_sync(0xffffffffu, hit);
        }
        if (!done) {  // the largest j of the sub-tile with w_j > 0 (rounding fallback)
            int best = -1;
            float wbest = 0.f;
#pragma unroll
            for (int e = 0; e < kW; ++e)
                if (wv[e] > 0.f) { best = j0 + e; wbest = wv[e]; }
            int jb = best;
            for (int o = 16; o > 0; o >>= 1) jb = max(jb, __shfl_xor_sync(0xffffffffu, jb, o));
            if (jb >= 0 && best == jb) {
                pick = jb;
                const float Wf = fix_to_float(W), tf = fix_to_float(tau);
                gap = fminf(Wf - tf, tf - (Wf - wbest)) / Wf;
            } else if (jb < 0 && lane == 0) {
                pick = e0 + tile * kSub;  // no positive entry: cannot happen when W > 0
            }
        }
    }
    if (pick >= 0) {
        out[depth] = pick;
        if (p.diag_gap) p.diag_gap[b] = gap;
    }
}

// ------------------------------------------------------------------ host
static bool tree_topology(const int32_t* parent, int n, TreeTopo* topo) {
    if (!parent || parent[0] != -1) return false;
    for (int i = 0; i < OSD_TREE_MAX_NODES; ++i) {
        topo->first_child[i] = -1;
        topo->next_sibling[i] = -1;
    }
    int8_t last_child[OSD_TREE_MAX_NODES];
    for (int i = 0; i < OSD_TREE_MAX_NODES; ++i) last_child[i] = -1;
    for (int i = 0; i < OSD_TREE_MAX_NODES; ++i) topo->parent[i] = -1;
    for (int i = 1; i < n; ++i) {
        const int par = parent[i];
        if (par < 0 || par >= i) return false;
        topo->parent[i] = static_cast<int8_t>(par);
        if (last_child[par] < 0) topo->first_child[par] = static_cast<int8_t>(i);
        else topo->next_sibling[last_child[par]] = static_cast<int8_t>(i);
        last_child[par] = static_cast<int8_t>(i);
    }
    return true;
}

static long long tree_stat_rows(int B, int n, bool greedy) { return (greedy ? 1LL : 2LL) * B * n; }

template <typename In>
static osd_status launch_tree(const TreeParams& base, int B, const void* draft, const void* target,
                              RowStat* stats, cudaStream_t stream) {
    TreeParams tp = base;
    const int n = tp.n, V = tp.V;
    constexpr size_t es = sizeof(In);
    if (tp.T == 0.f) {
        osd_status st = OSD_OK;
        int level[OSD_TREE_MAX_NODES] = {1}, depth = 1;  // rows of the longest walk
        for (int i = 1; i < n; ++i) depth = std::max(depth, level[i] = level[tp.topo.parent[i]] + 1);
        if (launch_greedy_walk<In>(GreedyTree{tp}, static_cast<const In*>(target), B, n, depth, V, stream, &st)) return st;
        const long long rows = tree_stat_rows(B, n, true);
        const int slice_len = stats_slice_len(rows);
        tp.n_slices = (V + slice_len - 1) / slice_len;
        tp.stats = stats;
        if (rows * tp.n_slices > INT_MAX) return OSD_ERR_UNSUPPORTED;
        const cudaError_t e = launch_ex(true, row_argmax_kernel<In>, dim3(unsigned(rows * tp.n_slices)), dim3(kStatThreads), 0, stream,
                                     1, static_cast<const In*>(target), V, slice_len, tp.n_slices, stats);
        if (e != cudaSuccess) return OSD_ERR_CUDA;
        return from_cuda(launch_ex(true, tree_greedy_kernel, dim3(unsigned(B)), dim3(kGreedyThreads), 0, stream, 1, tp));
    }
    // CTAs per sequence: 8, but 4 where 8 would run past one wave (two CTAs an SM) and the
    // spans stay short (B = 48 and 64 at V = 32000: 30.7 and 36.6 us against 39.7 and 44.9; at
    // V = 64000, B = 64 55.6 against 52.5)
    int c = kSeqMaxCluster;
    if ((long long)B * c > 2LL * device_sms() && V <= 50000) c /= 2;
    while (c > 1 && V <= 2048 * c) c /= 2;
    tp.span = ((V + c - 1) / c + 63) / 64 * 64;
    tp.csize = (V + tp.span - 1) / tp.span;
    if ((long long)B * tp.csize > INT_MAX) return OSD_ERR_UNSUPPORTED;
    // Nodes per round, by the bytes of one node of the batch: a round costs about 3 us beside
    // them, and first children that the walk does not come to are read for nothing (B = 1,
    // V = 32000: 4 nodes 14.2 us, 1 node 18.4; B = 32: 24.8, 2 nodes 23.1, 1 node 25.3; B = 64,
    // V = 128256, 33 MB: 2 nodes 85, 4 nodes 93, 1 node 83; B = 64, V = 150016 fp32, 77 MB: 1 node 134, 2
    // nodes 150).  A tree without siblings passes them often (B = 32, 9 nodes: 4 nodes 19.6 us, 2 21.3).
    const double pos = double(B) * 2 * V * double(es);
    bool siblings = false;
    for (int i = 0; i < n; ++i) siblings |= tp.topo.next_sibling[i] >= 0;
    const int win = pos <= 3e6 || (!siblings && pos <= 40e6) ? kTreeMaxWin : (pos <= 40e6 ? 2 : 1);
    const dim3 grid(unsigned(B) * unsigned(tp.csize));
    constexpr int sub = 32 * Elem<In>::kVec;
    const size_t smem = size_t((tp.span + sub - 1) / sub) * sizeof(float);
    const bool aligned = aligned_to(draft, 16) && aligned_to(target, 16) && ((size_t)V * es) % 16 == 0;
    return from_cuda(aligned ? launch_ex(true, tree_walk_kernel<In, true>, grid, dim3(kTreeThreads), smem, stream, tp.csize, tp, win)
                             : launch_ex(true, tree_walk_kernel<In, false>, grid, dim3(kTreeThreads), smem, stream, tp.csize, tp, win));
}

}  // namespace osd

extern "C" osd_status osd_verify_tree_workspace_size(int B, int n_nodes, int V, size_t* bytes) {
    using namespace osd;
    if (!bytes || B < 0 || n_nodes < 1 || V < 1) return OSD_ERR_INVALID_ARG;
    if (n_nodes > OSD_TREE_MAX_NODES || V > OSD_VERIFY_MAX_V) return OSD_ERR_UNSUPPORTED;
    const long long rows = tree_stat_rows(B, n_nodes, false);
    const int len = stats_slice_len(rows);
    // the greedy pass has half the rows but may take shorter slices: size for the larger
    const int len0 = stats_slice_len(tree_stat_rows(B, n_nodes, true));
    const size_t need = std::max(size_t(rows) * size_t((V + len - 1) / len),
                                 size_t(tree_stat_rows(B, n_nodes, true)) * size_t((V + len0 - 1) / len0)) *
                        sizeof(RowStat);
    *bytes = (need + 255) / 256 * 256;
    return OSD_OK;
}

extern "C" osd_status osd_verify_tree(const void* draft_logits, const void* target_logits, osd_dtype dtype, int B,
                                      int n_nodes, int V, const int32_t* parent, const int32_t* tokens,
                                      const float* uniforms, float temperature, int32_t* accepted, int32_t* path,
                                      int32_t* out_tokens, int32_t* last_node, float* diag_margin,
                                      float* diag_cdf_gap, void* workspace, size_t workspace_bytes, void* stream) {
    using namespace osd;
    if (dtype != OSD_F32 && dtype != OSD_BF16) return OSD_ERR_INVALID_ARG;
    if (B < 0 || n_nodes < 1 || V < 1) return OSD_ERR_INVALID_ARG;
    if (!(temperature >= 0.f) || !std::isfinite(temperature)) return OSD_ERR_INVALID_ARG;
    if (n_nodes > OSD_TREE_MAX_NODES || V > OSD_VERIFY_MAX_V) return OSD_ERR_UNSUPPORTED;
    TreeParams tp = {};
    if (!tree_topology(parent, n_nodes, &tp.topo)) return OSD_ERR_INVALID_ARG;
    if (B == 0) return OSD_OK;
    const bool greedy = (temperature == 0.f);
    const size_t es = dtype_size(dtype);
    if (!target_logits || !tokens || !accepted || !path || !out_tokens || !last_node || !workspace)
        return OSD_ERR_INVALID_ARG;
    if (!greedy && (!draft_logits || !uniforms)) return OSD_ERR_INVALID_ARG;
    if (!aligned_to(target_logits, es) || (draft_logits && !aligned_to(draft_logits, es)) ||
        !aligned_to(workspace, 16))
        return OSD_ERR_INVALID_ARG;
    size_t need = 0;
    osd_verify_tree_workspace_size(B, n_nodes, V, &need);
    if (workspace_bytes < need) return OSD_ERR_INVALID_ARG;
    tp.draft = draft_logits;
    tp.target = target_logits;
    tp.n = n_nodes;
    tp.V = V;
    tp.tokens = tokens;
    tp.uniforms = uniforms;
    tp.T = temperature;
    if (!greedy) split_scale(temperature, &tp.c_hi, &tp.c_lo);
    tp.accepted = accepted;
    tp.path = path;
    tp.out_tokens = out_tokens;
    tp.last_node = last_node;
    tp.diag_margin = diag_margin;
    tp.diag_gap = diag_cdf_gap;
    RowStat* stats = static_cast<RowStat*>(workspace);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    // the draft rows are not read at T = 0; any aligned pointer stands in
    const void* draft = greedy ? target_logits : draft_logits;
    return dtype == OSD_BF16 ? launch_tree<__nv_bfloat16>(tp, B, draft, target_logits, stats, s)
                             : launch_tree<float>(tp, B, draft, target_logits, stats, s);
}
