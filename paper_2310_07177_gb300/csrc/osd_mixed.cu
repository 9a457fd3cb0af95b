// osd_mixed.cu -- mixed-token sampling (Section 4.1 of the paper): one draw
// per position from beta p + (1 - beta) q_theta, p = softmax(t / tau),
// q = softmax(z / tau), by inverse CDF in ascending vocabulary order,
// j* = min{ j : C_j > u W } (the convention of the verifier's extra token).
//
// One CTA of kWarps warps per row, streaming both rows straight from HBM with
// 16-byte loads (one step of loads in flight ahead), no staging:
//
//   pass    every warp owns a contiguous part of the row and splits its steps
//           into kPieces runs; each lane keeps, per run, the online max and sum of
//           2^((x - max) c) of both rows, and the warp merges them at the end of
//           the run: 32 pieces of the CDF per row with 4 warps, 256 with 32;
//   pick    one warp merges the pieces into both normalisers, scans the piece
//           masses in fp64 for the piece that holds u W, and re-reads that one
//           piece to find the entry.
//
// Each logit is read once (plus one piece per row).  Small CTAs capped at 32
// registers a thread keep 16 rows (64 warps) in flight on every SM, and the
// single-warp pick of one row overlaps the streaming of the others; with few rows
// wider CTAs take over.  16384 x 32000 bf16 353 us, 87 % of the measured copy
// bandwidth; 16384 x 32001, off the 16-byte grid, 381 us (1021 us entry by entry).
#include <climits>
#include <type_traits>
#include <cmath>
#include <cstdint>

#include "osd.h"
#include "osd_device.cuh"
#include "osd_host.hpp"

namespace osd {

constexpr int kPieces = 8;  // runs per warp; a row of 4 warps has 32 pieces, one per lane of the picker

struct MixParams {
    const void* draft;
    const void* target;
    int V;
    long long dstride, tstride;  // elements between consecutive rows
    const float* uniforms;
    float beta;
    float c;  // log2(e) / tau, rounded to fp32
    int32_t* tokens;
    float* cdf_gap;
};

// Online sums of both rows over one piece, each as (M, s) with M = rn(max c)
// and s = sum 2^(x c - M).
struct Piece {
    float Mt, st, Mz, sz;
};

// How the rows lie: on 16-byte boundaries; off them, but both rows of a pair at the same
// place in a 16-byte vector (contiguous tensors of an odd vocabulary), so that chunks
// cut there are aligned in both; or anyhow, each chunk shifted into place from two
// aligned vectors.
constexpr int kMixAligned = 0, kMixPhased = 1, kMixShifted = 2;

template <typename In, int kMode, int kWarps>
__global__ void __launch_bounds__(32 * kWarps, 64 / kWarps) mixed_sample_kernel(MixParams p) {
    using E = Elem<In>;
    constexpr int kPer = kWarps * kPieces / 32;  // pieces per lane of the picker
    static_assert(kPer * 32 == kWarps * kPieces, "every lane holds as many pieces");
    constexpr int kW = E::kVec;  // entries per chunk
    __shared__ Piece s_piece[kWarps * kPieces];

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    grid_dependency_sync();
    const long long row = blockIdx.x;
    const In* zrow = static_cast<const In*>(p.draft) + row * p.dstride;
    const In* trow = static_cast<const In*>(p.target) + row * p.tstride;
    const int V = p.V;
    const float c = p.c;
    // chunk ci holds entries ci kW - ph ..
    const int ph = kMode == kMixPhased ? static_cast<int>((reinterpret_cast<uintptr_t>(zrow) & 15u) / sizeof(In)) : 0;
    // chunks of the row, the warp ranges and the runs (pieces) of steps in them
    const int nch = (V + ph + kW - 1) / kW;
    const int rch = (nch + kWarps - 1) / kWarps;  // chunks per warp range
    const int steps = (rch + 31) / 32;                   // steps of 32 chunks per range
    const int per_piece = (steps + kPieces - 1) / kPieces;
    auto range_lo = [&](int w) { return min(nch, w * rch); };

    // the kW raw entries of a chunk (outside the row they read as -inf)
    auto load_chunk = [&](const In* rp, int ci) -> uint4 {
        if constexpr (kMode == kMixAligned) {
            if ((ci + 1) * kW <= V) return ldg_stream(rp + size_t(ci) * kW);
        } else if constexpr (kMode == kMixPhased) {
            if (ci * kW >= ph && (ci + 1) * kW - ph <= V) return ldg_stream(rp + (ci * kW - ph));
        } else {
            if ((ci + 1) * kW <= V && shifted_inside(rp, ci * kW, V)) return ldg_shifted(rp + ci * kW);
        }
        float v[kW];  // the ragged first or last chunk of the row
#pragma unroll
        for (int e = 0; e < kW; ++e) {
            if constexpr (kMode == kMixPhased) {
                const int j = ci * kW - ph + e;
                v[e] = (j >= 0 && j < V) ? E::load(rp + j) : kNegInf;
            } else {
                v[e] = (ci * kW + e < V) ? E::load(rp + ci * kW + e) : kNegInf;
            }
        }
        return pack_raw<In, kW>(v);
    };
    const uint4 none = ninf_raw<In>();
    auto chunk_max = [](const uint4& r) { return E::max_raw(r); };
    // Exponent arguments are x c - M as one FMA, M = rn(m c): the FMA rounds
    // once, after the cancellation, so the terms that carry the mass come out
    // as exact as from the difference (x - m) c, and the rounding of M is a
    // factor common to all the sums it scales.  Rescaling between two
    // references is 2^(M - M'), a difference of two floats.
    auto chunk_sum = [&](const uint4& r, float M) {
        float x[kW];
        unpack_raw<In, kW>(r, x);
        float2 s2 = f2(0.f);
#pragma unroll
        for (int e = 0; e < kW; e += 2) {
            const float2 g = fma2(make_float2(x[e], x[e + 1]), f2(c), f2(-M));
            s2 = add2(s2, make_float2(ex2(g.x), ex2(g.y)));
        }
        return s2.x + s2.y;
    };
    // one lane's running (reference M, sum s) absorbs a chunk: rescale when the
    // reference rises (rarely, once the first chunks are in), then add; a lane
    // that has seen only -inf keeps s = 0 and skips the sum
    auto absorb = [&](float& M, float& s, const uint4& r) {
        const float cM = __fmul_rn(chunk_max(r), c);
        if (cM > M) {
            s = (M == kNegInf) ? 0.f : s * ex2(M - cM);
            M = cM;
        }
        if (M != kNegInf) s += chunk_sum(r, M);
    };
    // the warp's merge of every lane's (M, s); M = -inf marks a lane without mass
    auto warp_merge = [&](float& M, float& s) {
        float gM = M;
        for (int o = 16; o > 0; o >>= 1) gM = fmaxf(gM, __shfl_xor_sync(0xffffffffu, gM, o));
        s = (M == kNegInf) ? 0.f : s * ex2(M - gM);
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        M = gM;
    };

    // ---- pass: the warp's steps, one step of loads in flight ahead
    {
        const int c0 = range_lo(warp), c1 = range_lo(warp + 1);
        auto chunk_of = [&](int st) { return c0 + st * 32 + lane; };
        uint4 zc = none, tc = none;
        if (steps > 0 && chunk_of(0) < c1) {
            zc = load_chunk(zrow, chunk_of(0));
            tc = load_chunk(trow, chunk_of(0));
        }
        for (int g = 0; g < kPieces; ++g) {
            float Mt = kNegInf, st_ = 0.f, Mz = kNegInf, sz = 0.f;
            const int s_end = min((g + 1) * per_piece, steps);
            for (int st = g * per_piece; st < s_end; ++st) {
                uint4 zn = none, tn = none;
                if (st + 1 < steps && chunk_of(st + 1) < c1) {
                    zn = load_chunk(zrow, chunk_of(st + 1));
                    tn = load_chunk(trow, chunk_of(st + 1));
                }
                absorb(Mt, st_, tc);
                absorb(Mz, sz, zc);
                zc = zn;
                tc = tn;
            }
            warp_merge(Mt, st_);
            warp_merge(Mz, sz);
            if (lane == 0) s_piece[warp * kPieces + g] = Piece{Mt, st_, Mz, sz};
        }
    }
    __syncthreads();
    if (warp != 0) return;

    // ---- pick: lane l holds the pieces from kPer l (in vocabulary order)
    auto piece_of = [&](int i) { return s_piece[kPer == 1 ? lane : lane * kPer + i]; };
    const Piece first = piece_of(0);
    float Gt = first.Mt, Gz = first.Mz;  // rn(row max c): rounding is monotone, so the max of the M
#pragma unroll
    for (int i = 1; i < kPer; ++i) {
        Gt = fmaxf(Gt, piece_of(i).Mt);
        Gz = fmaxf(Gz, piece_of(i).Mz);
    }
    for (int o = 16; o > 0; o >>= 1) {
        Gt = fmaxf(Gt, __shfl_xor_sync(0xffffffffu, Gt, o));
        Gz = fmaxf(Gz, __shfl_xor_sync(0xffffffffu, Gz, o));
    }
    // each piece's sums against the row references (a piece of -inf only has none)
    float rt[kPer], rz[kPer];
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
        const Piece pc = i == 0 ? first : piece_of(i);
        rt[i] = (pc.Mt == kNegInf) ? 0.f : pc.st * ex2(pc.Mt - Gt);
        rz[i] = (pc.Mz == kNegInf) ? 0.f : pc.sz * ex2(pc.Mz - Gz);
    }
    float Et = rt[0], Ez = rz[0];
#pragma unroll
    for (int i = 1; i < kPer; ++i) {
        Et += rt[i];
        Ez += rz[i];
    }
    for (int o = 16; o > 0; o >>= 1) {
        Et += __shfl_xor_sync(0xffffffffu, Et, o);
        Ez += __shfl_xor_sync(0xffffffffu, Ez, o);
    }
    // weights w_j = a 2^(t_j c - G_t) + b 2^(z_j c - G_z) against the row references
    const float a = (Et > 0.f) ? p.beta / Et : 0.f;
    const float b = (Ez > 0.f) ? (1.f - p.beta) / Ez : 0.f;
    double mass = double(a) * double(rt[0]) + double(b) * double(rz[0]);
#pragma unroll
    for (int i = 1; i < kPer; ++i) mass += double(a) * double(rt[i]) + double(b) * double(rz[i]);
    const double incl = warp_incl_scan_f64(mass);
    const double W = __shfl_sync(0xffffffffu, incl, 31);
    const double tau = double(p.uniforms[row]) * W;
    int mode = 0, piece;  // mode 0: inverse CDF; 1: the largest j with w_j > 0
    double run = 0.0;
    const unsigned h = __ballot_sync(0xffffffffu, incl - mass <= tau && incl > tau);
    if (h) {
        piece = __ffs(h) - 1;
        run = __shfl_sync(0xffffffffu, incl - mass, piece);
        if constexpr (kPer > 1) {  // among that lane's pieces, the last one unless an earlier one passes tau
            int at = 0;
            double c2 = incl - mass;
#pragma unroll
            for (int i = 0; i < kPer - 1; ++i) {
                const double m = double(a) * double(rt[i]) + double(b) * double(rz[i]);
                if (at == i && c2 + m <= tau) {
                    c2 += m;
                    at = i + 1;
                }
            }
            run = __shfl_sync(0xffffffffu, c2, piece);
            piece = piece * kPer + __shfl_sync(0xffffffffu, at, piece);
        }
    } else if constexpr (kPer == 1) {
        mode = 1;
        const unsigned pos = __ballot_sync(0xffffffffu, mass > 0.0);
        piece = pos ? 31 - __clz(pos) : 0;
    } else {
        mode = 1;
        int last = -1;
#pragma unroll
        for (int i = 0; i < kPer; ++i)
            if (double(a) * double(rt[i]) + double(b) * double(rz[i]) > 0.0) last = lane * kPer + i;
        for (int o = 16; o > 0; o >>= 1) last = max(last, __shfl_xor_sync(0xffffffffu, last, o));
        piece = max(last, 0);
    }
    // a row without mass: its logits are -inf, and so are x c - 0
    const float Gt_ref = (Gt == kNegInf) ? 0.f : Gt, Gz_ref = (Gz == kNegInf) ? 0.f : Gz;
    const int pw = piece / kPieces, pg = piece % kPieces;
    const int c0 = range_lo(pw), c1 = range_lo(pw + 1);
    const int s_end = min((pg + 1) * per_piece, steps);
    int pick = -1, last_pos = -1;
    double gap = 0.0;
    bool found = false;
    for (int st = pg * per_piece; st < s_end; ++st) {  // warp-uniform trip count
        const int ci = c0 + st * 32 + lane;
        float z[kW], t[kW], w[kW];
        unpack_raw<In, kW>(ci < c1 ? load_chunk(zrow, ci) : none, z);
        unpack_raw<In, kW>(ci < c1 ? load_chunk(trow, ci) : none, t);
#pragma unroll
        for (int e = 0; e < kW; ++e) {
            const float pt = ex2(fmaf(t[e], c, -Gt_ref));
            const float qz = ex2(fmaf(z[e], c, -Gz_ref));
            w[e] = fmaf(a, pt, b * qz);
            if (w[e] > 0.f) last_pos = ci * kW - ph + e;
        }
        double mine = 0.0;
#pragma unroll
        for (int e = 0; e < kW; ++e) mine += double(w[e]);
        const double wincl = warp_incl_scan_f64(mine);
        if (mode == 0) {
            const double excl = run + wincl - mine;
            const unsigned hh = __ballot_sync(0xffffffffu, excl <= tau && excl + mine > tau);
            if (hh) {
                if (lane == __ffs(hh) - 1) {
                    double C = excl;
                    for (int e = 0; e < kW; ++e) {
                        const double Cprev = C;
                        C += double(w[e]);
                        if (C > tau) {
                            pick = ci * kW - ph + e;
                            gap = fmin(C - tau, tau - Cprev) / W;
                            break;
                        }
                    }
                    if (pick < 0) {  // the lane's entries pass tau only after rounding
                        pick = last_pos;
                        gap = 0.0;
                    }
                }
                found = true;
            }
        }
        if (found) break;
        run += __shfl_sync(0xffffffffu, wincl, 31);
    }
    if (!found) {  // mode 1, or rounding left tau past the piece: the largest j with w_j > 0
        int lp = last_pos;
        for (int o = 16; o > 0; o >>= 1) lp = max(lp, __shfl_xor_sync(0xffffffffu, lp, o));
        if (lane == 0) {
            pick = (lp >= 0) ? lp : (kMode == kMixPhased ? max(0, c0 * kW - ph) : c0 * kW);
            gap = (mode == 1) ? (W - tau) / W : 0.0;
        }
    }
    if (pick >= 0) {
        p.tokens[row] = pick;
        if (p.cdf_gap) p.cdf_gap[row] = float(gap);
    }
}

}  // namespace osd

extern "C" osd_status osd_mixed_sample(const void* draft_logits, const void* target_logits, osd_dtype dtype, int N,
                                       int V, int64_t d_stride, int64_t t_stride, const float* uniforms, float beta,
                                       float temperature, int32_t* tokens, float* cdf_gap, int32_t* status,
                                       void* stream) {
    using namespace osd;
    if (dtype != OSD_F32 && dtype != OSD_BF16) return OSD_ERR_INVALID_ARG;
    if (N < 0 || V < 1 || d_stride < 0 || t_stride < 0) return OSD_ERR_INVALID_ARG;
    if (!(beta >= 0.f && beta <= 1.f)) return OSD_ERR_INVALID_ARG;
    if (!(temperature > 0.f) || !std::isfinite(temperature)) return OSD_ERR_INVALID_ARG;
    if (V > OSD_VERIFY_MAX_V) return OSD_ERR_UNSUPPORTED;
    const size_t es = dtype_size(dtype);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (status && !aligned_to(status, 4)) return OSD_ERR_INVALID_ARG;
    if (status) {  // no wait in this kernel can run out: the status is OSD_OK once the launch is queued
        const cudaError_t e = cudaMemsetAsync(status, 0, sizeof(int32_t), s);
        if (e != cudaSuccess) return OSD_ERR_CUDA;
    }
    if (N == 0) return OSD_OK;
    if (!draft_logits || !target_logits || !uniforms || !tokens) return OSD_ERR_INVALID_ARG;
    if (!aligned_to(draft_logits, es) || !aligned_to(target_logits, es) || !aligned_to(uniforms, 4) ||
        !aligned_to(tokens, 4) || (cdf_gap && !aligned_to(cdf_gap, 4)))
        return OSD_ERR_INVALID_ARG;
    auto row_ok = [&](int64_t stride) { return N <= 1 || (stride * int64_t(es)) % 16 == 0; };
    const bool vec = aligned_to(draft_logits, 16) && aligned_to(target_logits, 16) && row_ok(d_stride) &&
                     row_ok(t_stride);
    const bool phased = (reinterpret_cast<uintptr_t>(draft_logits) - reinterpret_cast<uintptr_t>(target_logits)) % 16 == 0 &&
                        row_ok(d_stride - t_stride);
    MixParams mp;
    mp.draft = draft_logits;
    mp.target = target_logits;
    mp.V = V;
    mp.dstride = d_stride;
    mp.tstride = t_stride;
    mp.uniforms = uniforms;
    mp.beta = beta;
    mp.c = static_cast<float>(1.4426950408889634074 / static_cast<double>(temperature));
    mp.tokens = tokens;
    mp.cdf_gap = cdf_gap;
    // Warps per row: 4, 64 warps an SM over many rows, but 16 or 32 where so few rows leave the
    // SMs idle and a warp then still has a few steps (of 32 chunks) of its own; very long rows
    // do better with 32 up to one wave of 4-warp rows.  In us, 4 / 16 / 32 warps (bf16): 100 x 32000
    // 22.6 / 13.0 / 14.5, 600 x 32000 34.4 / 28.7 / 37.8, 1000 x 32000 39.5 / 44.7 / 60.1,
    // 20 x 5000 9.3 / 9.8 / 12.3, 300 x 128256 111 / 47 / 39, 1000 x 128256 130 / 129 / 113,
    // 4096 x 128257 406 / 386 / 427; fp32, 1 x 75651 56 / 25 / 20.
    const int sms = device_sms();
    auto go_warps = [&](auto tag, auto mode) {
        using In = decltype(tag);
        constexpr int kMode = decltype(mode)::value;
        const dim3 grid(static_cast<unsigned>(N));
        const int steps = V / (32 * Elem<In>::kVec);
        const int ww = steps > 256 && N <= (steps > 400 ? 16 : 4) * sms ? 32 : (steps > 24 && N <= (steps > 64 ? 4 : 2) * sms ? 16 : 4);
        // a start before the previous kernel's end packs a call that fills the SMs onto those that
        // become free first (1761 x 16256: 36.7 us against 34.0 without; 50 x 32000: 10.1 against 12.3)
        const bool early = N <= sms;
        if (ww == 32) return launch_ex(early, mixed_sample_kernel<In, kMode, 32>, grid, dim3(1024), 0, s, 1, mp);
        if (ww == 16) return launch_ex(early, mixed_sample_kernel<In, kMode, 16>, grid, dim3(512), 0, s, 1, mp);
        return launch_ex(early, mixed_sample_kernel<In, kMode, 4>, grid, dim3(128), 0, s, 1, mp);
    };
    auto go = [&](auto tag) {
        if (vec) return go_warps(tag, std::integral_constant<int, kMixAligned>());
        if (phased) return go_warps(tag, std::integral_constant<int, kMixPhased>());
        return go_warps(tag, std::integral_constant<int, kMixShifted>());
    };
    const cudaError_t e = dtype == OSD_BF16 ? go(__nv_bfloat16()) : go(float());
    return from_cuda(e);
}
