// pps_misc.cu -- detector pass, raw keyed words, and the fp32 key self-test.
#include <climits>
#include <cstdint>

#include "pps_device.cuh"
#include "pps_internal.h"

namespace pps {

#define FULL 0xffffffffu

// Detector (App. E): every warp takes a contiguous chunk of tokens and works
// through it a group of 128 at a time; lane l loads and scores tokens 2l,
// 2l + 1, 64 + 2l and 65 + 2l of the group (whole lines per load when the arrays are
// aligned), the four Philox blocks round by round side by side.  When the whole group has one key
// (the tokens of one text), the key schedule is warp-uniform and kept in
// uniform registers.  Segment sums: the warp keeps a window of 32 segment
// starts, one per lane, and finds a group's segments by a ballot; a group of up
// to kSegRounds segments takes one masked warp reduction per segment, one of
// more is rearranged to lane-major order (shuffles) and takes a segmented warp
// scan per 32 tokens.  The running sum of the open segment is a
// float-float pair (an exact fp32 two-sum per addition, FP64 being slow on this
// part) and goes to the segment's fp64 slot with one atomic per segment end the
// warp sees (plus one at the end of its chunk).
//
// 10^7 tuples (280 MB with the scores): about 62 us = 4.5 TB/s, 0.66 of the measured copy rate, the segment
// pass 17 us; 10^7 tuples in texts of 128 took 96.5 us with their p-values and take 86, 6.6 10^6
// in ragged texts of 400 tokens 130 and 90.  The kernel issues 130 instructions a tuple (40 of them the Philox
// block) in 55% of its cycles; copying the next group's inputs to shared memory ahead (86 us),
// five CTAs an SM of 48 registers (86 us) and sending finished sums 32 at a time (90 and 90 us before
// the segment pass was split) changed nothing.
constexpr int kScoreAhead = 4;  // tuples per lane of a group
constexpr int kSegRounds = 6;

// hi + lo += v, with the rounding error of hi + v kept in lo (two-sum)
__device__ __forceinline__ void ff_add(float& hi, float& lo, float v) {
    const float s = hi + v;
    const float bp = s - hi;
    lo += (hi - (s - bp)) + (v - bp);
    hi = s;
}

// The first-arrival words of a lane's four tuples; UNI: under one key that the
// whole warp holds (from warp reductions, so its schedule stays in uniform registers).
template <bool UNI>
__device__ __forceinline__ void words4(const int32_t (&tk)[4], const uint64_t (&kk)[4], const uint64_t (&cx)[4],
                                       const uint32_t (&ps)[4], uint32_t klo, uint32_t khi, uint32_t (&w)[4]) {
    uint32_t x0[4], x1[4], x2[4], x3[4], k0[4], k1[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        x0[u] = (uint32_t)((uint64_t)(int64_t)tk[u] >> 2);
        x1[u] = ps[u];
        x2[u] = (uint32_t)cx[u];
        x3[u] = (uint32_t)(cx[u] >> 32);
        k0[u] = UNI ? klo : (uint32_t)kk[u];
        k1[u] = UNI ? khi : (uint32_t)(kk[u] >> 32);
    }
#pragma unroll
    for (int r = 0; r < PPS_PHILOX_ROUNDS; ++r) {
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            uint32_t hi0, lo0, hi1, lo1;
            mulhilo(kPhiloxM0, x0[u], hi0, lo0);
            mulhilo(kPhiloxM1, x2[u], hi1, lo1);
            x0[u] = hi1 ^ x1[u] ^ (k0[u] + (uint32_t)r * kPhiloxW0);
            x2[u] = hi0 ^ x3[u] ^ (k1[u] + (uint32_t)r * kPhiloxW1);
            x1[u] = lo1;
            x3[u] = lo0;
        }
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) w[u] = lane_of(make_uint4(x0[u], x1[u], x2[u], x3[u]), (uint32_t)(tk[u] & 3));
}

template <bool VEC>
__global__ void __launch_bounds__(256, 4) wm_score_kernel(const int32_t* __restrict__ tokens,
                                                       const uint64_t* __restrict__ key,
                                                       const uint64_t* __restrict__ ctx,
                                                       const uint32_t* __restrict__ pos, int64_t n, int32_t n_seg,
                                                       const int64_t* __restrict__ seg_off, ScoreParams P,
                                                       float* out_score, double* out_sum, int64_t chunk) {
    const int lane = threadIdx.x & 31;
    const int64_t gw = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t c0 = gw * chunk;
    if (c0 >= n) return;
    const int64_t c1 = min(n, c0 + chunk);
    const bool segs = out_sum != nullptr && seg_off != nullptr;
    // the open segment (warp-uniform) and its end; win: the start of segment wb + lane
    int seg = 0, wb = 0;
    int64_t seg_end = LLONG_MAX, win = LLONG_MAX;
    // open the last segment that starts at or before t (from the window on)
    auto open_segment = [&](int64_t t) {
        while (true) {
            const int m = __popc(__ballot_sync(FULL, win <= t));
            if (m < 32) {
                seg = wb + max(m, 1) - 1;
                seg_end = __shfl_sync(FULL, win, max(m, 1));
                return;
            }
            wb += 31;
            win = wb + lane < n_seg ? seg_off[wb + lane] : LLONG_MAX;
        }
    };
    if (segs) {
        // 32 probes a step: seg_off[wb] <= c0 < seg_off[hi]
        int hi = n_seg;
        while (hi - wb > 32) {
            const int step = (hi - wb + 31) / 32;
            const int64_t at = (int64_t)wb + (int64_t)lane * step;
            const int m = __popc(__ballot_sync(FULL, at < hi && seg_off[at] <= c0));
            wb += (max(m, 1) - 1) * step;
            hi = min(hi, wb + step);
        }
        win = wb + lane < n_seg ? seg_off[wb + lane] : LLONG_MAX;
        open_segment(c0);
    }
    float chi = 0.0f, clo = 0.0f;  // running sum of the open segment
    auto flush = [&]() {
        if (lane == 0 && (chi != 0.0f || clo != 0.0f)) atomicAdd(out_sum + seg, (double)chi + (double)clo);
        chi = clo = 0.0f;
    };
    constexpr int G = 32 * kScoreAhead;
    static_assert(kScoreAhead == 4, "a lane holds four tuples of a group");
    for (int64_t grp = c0; grp < c1; grp += G) {
        // lane l holds tuples grp + 2 l, 2 l + 1, 64 + 2 l and 65 + 2 l (bits of `on`: those that
        // exist), so that every load and store of the warp covers whole lines
        const int64_t t0 = grp + 2 * lane;
        const int nleft = (int)min((int64_t)G, c1 - grp);
        const unsigned on = nleft == G ? 0xfu
                                       : (unsigned)(2 * lane < nleft) | ((unsigned)(2 * lane + 1 < nleft) << 1) |
                                             ((unsigned)(2 * lane + 64 < nleft) << 2) | ((unsigned)(2 * lane + 65 < nleft) << 3);
        int32_t tk[4] = {0, 0, 0, 0};
        uint64_t kk[4] = {0, 0, 0, 0}, cx[4] = {0, 0, 0, 0};
        uint32_t ps[4] = {0, 0, 0, 0};
        if (VEC && nleft == G) {
            const int2 ta = __ldg(reinterpret_cast<const int2*>(tokens + t0)), tb = __ldg(reinterpret_cast<const int2*>(tokens + t0 + 64));
            const uint2 pa = __ldg(reinterpret_cast<const uint2*>(pos + t0)), pb = __ldg(reinterpret_cast<const uint2*>(pos + t0 + 64));
            const ulonglong2 ka = __ldg(reinterpret_cast<const ulonglong2*>(key + t0));
            const ulonglong2 kb = __ldg(reinterpret_cast<const ulonglong2*>(key + t0 + 64));
            const ulonglong2 xa = __ldg(reinterpret_cast<const ulonglong2*>(ctx + t0));
            const ulonglong2 xb = __ldg(reinterpret_cast<const ulonglong2*>(ctx + t0 + 64));
            tk[0] = ta.x; tk[1] = ta.y; tk[2] = tb.x; tk[3] = tb.y;
            ps[0] = pa.x; ps[1] = pa.y; ps[2] = pb.x; ps[3] = pb.y;
            kk[0] = ka.x; kk[1] = ka.y; kk[2] = kb.x; kk[3] = kb.y;
            cx[0] = xa.x; cx[1] = xa.y; cx[2] = xb.x; cx[3] = xb.y;
        } else {
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if ((on >> u) & 1u) {
                    const int64_t t = t0 + (u & 1) + 64 * (u >> 1);
                    tk[u] = tokens[t];
                    ps[u] = pos[t];
                    kk[u] = key[t];
                    cx[u] = ctx[t];
                }
        }
        // one key for the whole group (the tokens of one text): its schedule in uniform registers
        const uint32_t klo = __reduce_or_sync(FULL, (uint32_t)kk[0]), khi = __reduce_or_sync(FULL, (uint32_t)(kk[0] >> 32));
        uint32_t odd = 0;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const uint32_t d = ((uint32_t)kk[u] ^ klo) | ((uint32_t)(kk[u] >> 32) ^ khi);
            odd |= (on >> u) & 1u ? d : 0u;
        }
        uint32_t w[4];
        if (__all_sync(FULL, odd == 0u)) words4<true>(tk, kk, cx, ps, klo, khi, w);
        else words4<false>(tk, kk, cx, ps, 0u, 0u, w);
        float A[4];
        if (P.kind == 0) {
#pragma unroll
            for (int u = 0; u < 4; ++u) A[u] = score32(w[u]);
        } else {
#pragma unroll
            for (int u = 0; u < 4; ++u) A[u] = score_kind32(w[u], P);
        }
        if (nleft < G) {
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (!((on >> u) & 1u)) A[u] = 0.0f;
        }
        if (out_score) {
            if (VEC && nleft == G) {
                *reinterpret_cast<float2*>(out_score + t0) = make_float2(A[0], A[1]);
                *reinterpret_cast<float2*>(out_score + t0 + 64) = make_float2(A[2], A[3]);
            } else {
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    if ((on >> u) & 1u) out_score[t0 + (u & 1) + 64 * (u >> 1)] = A[u];
            }
        }
        if (!out_sum) continue;
        const int64_t gend = min(grp + G, c1);
        if (segs && grp >= seg_end) {
            // the open segment ended before this group: flush it, open the group's first segment
            flush();
            open_segment(grp);
        }
        if (gend <= seg_end) {
            // the whole group lies in the open segment (or there is one segment)
            float v = (A[0] + A[1]) + (A[2] + A[3]);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(FULL, v, o);
            ff_add(chi, clo, v);
            continue;
        }
        // segments that start inside the group, as far as the window shows them
        const unsigned inside = __ballot_sync(FULL, win > grp && win < gend);
        if (__popc(inside) < kSegRounds && __shfl_sync(FULL, win, 31) >= gend) {
            // one masked reduction per segment of the group
            int64_t s0 = grp;
            while (true) {
                const int64_t s1 = min(seg_end, gend);
                const int a = (int)(s0 - grp), b = (int)(s1 - grp);
                float v = 0.0f;
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int at = 2 * lane + (u & 1) + 64 * (u >> 1);
                    v += at >= a && at < b ? A[u] : 0.0f;
                }
#pragma unroll
                for (int o = 16; o > 2; o >>= 1) v += __shfl_xor_sync(FULL, v, o);
                // the four sums of 32 are added without loss, as the scan below adds its sums of 32:
                // sums of up to 128 in fp32 alone left segments of 100 to 160 tokens a relative rms error
                // of 3.2e-8, these 1.9e-8, the scan 2.2e-8 (6.6 10^6 tuples in texts of 38: 215 -> 218 us)
                float lo = 0.0f;
#pragma unroll
                for (int o = 2; o > 0; o >>= 1) {
                    const float ov = __shfl_xor_sync(FULL, v, o);
                    if (o == 1) lo += __shfl_xor_sync(FULL, lo, o);
                    ff_add(v, lo, ov);
                }
                ff_add(chi, clo, v);
                clo += lo;
                if (seg_end >= gend) break;  // stays open
                s0 = seg_end;
                flush();
                open_segment(s0);
            }
            continue;
        }
        // many short segments: a segmented scan per iteration, over the
        // lane-major layout (iteration u, lane t: tuple grp + 32 u + t, pair (32 u + t) / 64 of
        // lane 16 (u mod 2) + t / 2)
        float Am[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int src = 16 * (u & 1) + (lane >> 1);
            const float a0 = __shfl_sync(FULL, A[u & 2], src), a1 = __shfl_sync(FULL, A[(u & 2) + 1], src);
            Am[u] = lane & 1 ? a1 : a0;
        }
#pragma unroll 1
        for (int u = 0; u < kScoreAhead; ++u) {
            const int64_t base = grp + 32 * u;
            if (base >= c1) break;
            const int64_t t = base + lane;
            // segment of my token, advanced from the warp's open segment (segments are contiguous)
            int my = INT_MAX;
            if (t < c1) {
                my = seg;
                while (my + 1 < n_seg && seg_off[my + 1] <= t) ++my;
            }
            // segmented inclusive scan over the lanes of each segment run
            float v = u == 0 ? Am[0] : u == 1 ? Am[1] : u == 2 ? Am[2] : Am[3];
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const float ov = __shfl_up_sync(FULL, v, o);
                const int os = __shfl_up_sync(FULL, my, o);
                if (lane >= o && os == my) v += ov;
            }
            // the open segment ended before this iteration's first run: flush it
            const int s0 = __shfl_sync(FULL, my, 0);
            if (s0 != seg) {
                flush();
                seg = s0;
            }
            const int nxt = __shfl_down_sync(FULL, my, 1);
            const bool more = base + 32 < c1;
            if (t < c1 && (lane == 31 || nxt != my)) {
                const bool open = lane == 31 && more;  // may continue into the next iteration
                if (!open) atomicAdd(out_sum + my, (double)v + (my == seg ? (double)chi + (double)clo : 0.0));
            }
            if (more) {
                const float v31 = __shfl_sync(FULL, v, 31);
                const int s31 = __shfl_sync(FULL, my, 31);
                if (s31 == seg) {
                    ff_add(chi, clo, v31);
                } else {
                    chi = v31;
                    clo = 0.0f;
                }
                seg = s31;
            } else {
                chi = clo = 0.0f;
            }
        }
        // the window from the open segment on
        wb = seg;
        win = wb + lane < n_seg ? seg_off[wb + lane] : LLONG_MAX;
        seg_end = __shfl_sync(FULL, win, 1);
    }
    // the chunk's open sum (the scan path flushes its own at the chunk's end)
    if (out_sum) flush();
}

// ln Gamma(x) for x >= 16 by Stirling's asymptotic series (truncation error
// below 1e-16 there); smaller x through the recurrence Gamma(x+1) = x Gamma(x).
__device__ double lgamma_stirling(double x) {
    double shift = 0.0;
    while (x < 16.0) {
        shift -= log(x);
        x += 1.0;
    }
    const double r = 1.0 / x, r2 = r * r;
    const double series = r * (1.0 / 12.0 - r2 * (1.0 / 360.0 - r2 * (1.0 / 1260.0 - r2 * (1.0 / 1680.0))));
    return shift + (x - 0.5) * log(x) - x + 0.91893853320467274178 + series;
}

// Stirling's series of ln Gamma(M) - (M - 1/2) ln M + M - ln sqrt(2 pi) for M >= 16
// (1/(12M) and its next three terms; below 1e-3 there, so fp32 suffices)
__device__ __forceinline__ float stirling_tail(float M) {
    const float r = 1.0f / M, r2 = r * r;
    return r * (1.0f / 12.0f - r2 * (1.0f / 360.0f - r2 * (1.0f / 1260.0f - r2 * (1.0f / 1680.0f))));
}

// ln of the Poisson term e^-S S^k / k! for k = M - 1 (top = false) or k = M (top = true).
// For M >= 16, with y = S/M - 1 and Stirling's formula for ln Gamma(M) (ln M! = ln Gamma(M)
// + ln M), both are k log1p(y) - (S - M) - ln sqrt(2 pi M) - stirling_tail(M): the large
// parts S and k ln S cancel against M and k ln M inside log1p, so one fp64 log1p is the
// only fp64 transcendental, and the M-only terms (below ~12) are fp32 (errors < 1e-6).
// Smaller M take ln Gamma from lgamma_stirling.
__device__ double poisson_lead(int64_t M, double S, bool top) {
    if (M < 16) {
        const double ls = log(S);
        return top ? -S + (double)M * ls - lgamma_stirling((double)M + 1.0)
                   : -S + (double)(M - 1) * ls - lgamma_stirling((double)M);
    }
    const double Md = (double)M;
    double rM = (double)(1.0f / (float)M);
    rM = rM * (2.0 - Md * rM);  // one Newton step: relative error ~1e-14
    const double y = (S - Md) * rM;
    const float Mf = (float)M;
    const float c = 0.5f * logf(6.28318530717958648f * Mf) + stirling_tail(Mf);
    return (top ? Md : Md - 1.0) * log1p(y) - (S - Md) - (double)c;
}

// The ratios r_m (r_0 = 1) of the Poisson terms to the leading one, summed in
// compensated (Kahan) fp32 until a term drops below 1e-12 of the sum: downward
// (S >= M: r_m = r_{m-1} (M - m) / S, s = 1/S in fp32) or upward (S < M:
// r_m = r_{m-1} S / (M + m), s = S in fp32).  Also returns sum_m m r_m, the
// first-order sensitivity to the relative error of s.  For M < kSeriesF64Min,
// where the counters are exact in fp32 (int64 -> fp32 conversions in the loop
// cost a quarter of the kernel).
template <bool DOWN>
__device__ __forceinline__ void poisson_ratios(int64_t M, float s, float& sum, float& wsum) {
    float r = 1.0f, comp = 0.0f, m = 0.0f;
    sum = 1.0f;
    wsum = 0.0f;
    for (float j = (float)(DOWN ? M - 1 : M + 1); !DOWN || j > 0.0f; j += DOWN ? -1.0f : 1.0f) {
        r *= DOWN ? j * s : s / j;
        m += 1.0f;
        const float y = r - comp, t = sum + y;
        comp = (t - sum) - y;
        sum = t;
        wsum = fmaf(m, r, wsum);
        if (r < 1e-12f * sum) break;
    }
}

// From this segment length on the series runs in fp64: with S near M, successive
// ratios j/S differ by ~1/M, below the fp32 spacing near 1 for M ~ 2^24, so their
// rounding errors stop averaging out and the fp32 product drifts (measured on the
// host: 7e-7 in ln p at M = 2^16, 1.3e-5 at 2^24).  Such segments are rare; their
// ~6 sqrt(M) fp64 steps cost microseconds.
constexpr int64_t kSeriesF64Min = 1 << 18;

// ln P(Gamma(M,1) >= S) for integer M >= 1, as the Poisson probability
// P(N <= M-1), N ~ Poisson(S).  The leading term e^-S S^j / j! at j = M-1
// (S >= M) or j = M (S < M) is taken in fp64 (poisson_lead); the sum of the
// ratios of the other terms to it, all <= 1 and summed away from the mode
// until they stop mattering: for S >= M downward from M-1 (ratios j/S), below
// as 1 - P(N >= M) upward from M (ratios S/j).  Below kSeriesF64Min tokens in
// compensated fp32 (poisson_ratios; FP64 throughput is low on this part) with a
// first-order correction for the fp32 image of S (the m-th term carries it m
// times: with its relative error d, the exact sum is sum + d * sum_m m r_m);
// error below 1e-6 absolute in ln p.  From kSeriesF64Min on in fp64.
//
// gamma_ratios: that corrected sum (fp32 series); gamma_from: ln P from it and
// the leading term.  The two parts do not depend on each other.
__device__ double gamma_ratios(int64_t M, double S) {
    const float Sf = (float)S;
    float sum, wsum;
    if (S >= (double)M) {
        const float inv = 1.0f / Sf;
        // d = (1/S) / inv - 1 = e / (1 - e) with e = 1 - S inv (|e| < 1e-7): e + e^2
        const double e = 1.0 - S * (double)inv;
        const double d = fma(e, e, e);
        poisson_ratios<true>(M, inv, sum, wsum);
        return (double)sum + d * (double)wsum;
    }
    const double d = (S - (double)Sf) * (double)(1.0f / Sf);  // relative error of Sf (its own error ~1e-14)
    poisson_ratios<false>(M, Sf, sum, wsum);
    return (double)sum + d * (double)wsum;
}
__device__ double gamma_from(int64_t M, double S, double lead, double tot) {
    // tot in [1, ~1e3]: its logarithm in fp32 errs by ~1e-7 absolute
    if (S >= (double)M) return lead + (double)logf((float)tot);
    // S < M: P(N >= M) <= ~1/2, so ln(1 - P(N >= M)) in fp32 errs by ~1e-7 absolute
    return (double)log1pf(-expf((float)lead) * (float)tot);
}
__device__ __noinline__ double gamma_tail_long(int64_t M, double S) {
    double r = 1.0, sum = 1.0;
    if (S >= (double)M) {
        const double inv = 1.0 / S;
        for (int64_t j = M - 1; j > 0; --j) {
            r *= (double)j * inv;
            sum += r;
            if (r < 1e-17 * sum) break;
        }
        return poisson_lead(M, S, false) + log(sum);
    }
    for (int64_t j = M + 1;; ++j) {
        r *= S / (double)j;
        sum += r;
        if (r < 1e-17 * sum) break;
    }
    return log1p(-exp(poisson_lead(M, S, true)) * sum);
}

// Chernoff bound on ln P(U_1 + ... + U_M >= S): the exponent
// M ln((e^l - 1)/l) - l S at the l where the mean of the exponentially tilted
// uniform, 1/(1 - e^-l) - 1/l, equals S/M (fp32 Newton steps kept inside a
// bisection bracket; the exponent is flat there, and is evaluated in fp64).
// 0 for S <= M/2, -inf for S >= M.
__device__ double chernoff_u_logp(int64_t M, double S) {
    const double x = S / (double)M;
    if (!(x > 0.5)) return 0.0;
    if (x >= 1.0) return -INFINITY;
    const float xf = (float)x;
    auto mean = [](float l) {
        if (l < 1e-2f) return 0.5f + l / 12.0f - l * l * l / 720.0f;
        return 1.0f / (-expm1f(-l)) - 1.0f / l;
    };
    auto slope = [](float l) {  // variance of the tilted uniform
        if (l < 1e-2f) return 1.0f / 12.0f - l * l / 240.0f;
        const float e = expf(-l), d = -expm1f(-l);
        return 1.0f / (l * l) - e / (d * d);
    };
    float lo = 0.0f, hi = 2.0f / (1.0f - xf) + 10.0f;
    float l = xf < 0.75f ? 12.0f * (xf - 0.5f) : 1.0f / (1.0f - xf);
    for (int it = 0; it < 60; ++it) {
        const float f = mean(l) - xf;
        if (f > 0.0f) hi = l;
        else lo = l;
        float nl = l - f / slope(l);
        if (!(nl > lo && nl < hi)) nl = 0.5f * (lo + hi);
        if (fabsf(nl - l) <= 1e-6f * l) {
            l = nl;
            break;
        }
        l = nl;
    }
    const double ld = (double)l;
    const double e = (double)M * log(expm1(ld) / ld) - ld * S;
    return e < 0.0 ? e : 0.0;
}

// per-segment ln p-values from the segment sums (kind 0 Gamma tail, 1 Chernoff on U).
// A CTA takes kLogpSegs segments; for the Gamma tail its second half of warps
// evaluates the leading terms (a chain of fp64) while the first half runs the fp32
// series of the same segments: each is a latency chain of about the same length
// (one thread for both: 16400 segments of 400 tokens 111 us with their scores, now 91).
constexpr int kLogpSegs = 64;
__global__ void __launch_bounds__(2 * kLogpSegs) seg_logp_kernel(int64_t n, int32_t n_seg,
                                                                  const int64_t* __restrict__ seg_off,
                                                                  const double* __restrict__ sums, int kind,
                                                                  double* out_logp) {
    __shared__ double s_lead[kLogpSegs];
    const int i = threadIdx.x % kLogpSegs;
    const bool second = threadIdx.x >= kLogpSegs;
    const int64_t g = (int64_t)blockIdx.x * kLogpSegs + i;
    int64_t M = 0;
    double S = 0.0;
    if (g < n_seg) {
        M = seg_off ? seg_off[g + 1] - seg_off[g] : n;
        S = sums[g];
    }
    const bool series = kind == 0 && M > 0 && M < kSeriesF64Min && S > 0.0;
    double tot = 1.0;
    if (series) {
        if (second) s_lead[i] = poisson_lead(M, S, !(S >= (double)M));
        else tot = gamma_ratios(M, S);
    }
    __syncthreads();
    if (second || g >= n_seg) return;
    double lp;
    if (series)
        lp = gamma_from(M, S, s_lead[i], tot);
    else if (M <= 0 || (kind == 0 && !(S > 0.0)))
        lp = 0.0;
    else if (kind == 0)
        lp = gamma_tail_long(M, S);
    else if (kind == 1)
        lp = chernoff_u_logp(M, S);
    else
        lp = __longlong_as_double(0x7ff8000000000000ll);  // NaN: no null law for this score
    out_logp[g] = lp;
}

// SplitMix64's output function (Steele, Lea, Flood, OOPSLA'14): the labeler of
// a child context, label(c || u) = mix(label(c) ^ (u + 1) * 0x9E3779B97F4A7C15)
__device__ __forceinline__ uint64_t mix64(uint64_t z) {
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

// One depth of the dynamic IID draft tree (layout in pps.h): warp b takes
// sequence b, lane i the depth's row i; the distinct labels of the present
// rows get consecutive child slots (exclusive scan over the rows).
__global__ void tree_expand_kernel(int32_t n_seq, int32_t K, int32_t gamma, int32_t depth,
                                   const int32_t* __restrict__ tok, const int32_t* __restrict__ mult,
                                   const int32_t* __restrict__ ndist, const uint64_t* __restrict__ key,
                                   const uint64_t* __restrict__ ctx, const uint32_t* __restrict__ pos,
                                   const int32_t* __restrict__ row_k, uint64_t* next_key, uint64_t* next_ctx,
                                   uint32_t* next_pos, int32_t* next_k, int32_t* child_node, uint64_t* node_key,
                                   uint64_t* node_ctx, uint32_t* node_pos) {
    pdl_wait();  // the lists and row ids of the previous launch
    pdl_launch_dependents();
    const int lane = threadIdx.x & 31;
    const int64_t b = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (b >= n_seq) return;
    const int64_t N1 = 1 + (int64_t)K * gamma;
    const int w = depth == 0 ? 1 : K;
    // draft rows are numbered depth-major: depth d's rows start at D_d = n_seq (1 + (d-1) K)
    const int64_t D_d = depth == 0 ? 0 : (int64_t)n_seq * (1 + (int64_t)(depth - 1) * K), off_n = 1 + (int64_t)depth * K;
    const int64_t r = b * w + lane;
    const bool row = lane < w;
    int nd = 0;
    if (row && row_k[r] > 0) nd = max(0, min(ndist[r], K));
    int j0 = nd;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(FULL, j0, o);
        if (lane >= o) j0 += t;
    }
    const int total = min(__shfl_sync(FULL, j0, 31), K);
    j0 -= nd;
    if (row) {
        const int64_t dr = D_d + b * w + lane;
        for (int m = 0; m < K; ++m) {
            int node = -1;
            const int j = j0 + m;
            if (m < nd && j < K) {
                const int64_t q = b * K + j;
                const uint64_t lab = mix64(ctx[r] ^ ((uint64_t)(uint32_t)(tok[r * K + m] + 1) * 0x9E3779B97F4A7C15ull));
                next_key[q] = key[r];
                next_ctx[q] = lab;
                next_pos[q] = pos[r] + 1u;
                next_k[q] = mult[r * K + m];
                node = (int)(b * N1 + off_n + j);
                node_key[node] = key[r];
                node_ctx[node] = lab;
                node_pos[node] = pos[r] + 1u;
            }
            child_node[dr * K + m] = node;
        }
    }
    for (int j = lane; j < K; j += 32)
        if (j >= total) {
            const int64_t q = b * K + j;
            next_key[q] = key[b * w];
            next_ctx[q] = 0;
            next_pos[q] = 0;
            next_k[q] = 0;
        }
}

// One depth of the draft tree of B non-identical proposals (layout in pps.h):
// warp s takes sequence s, lane b proposal b.  A proposal at node o of depth
// d that drew token x moves to child (d+1, f), f = the first proposal at the
// same node that drew x; node o's list holds the distinct tokens of its
// proposals in proposal order, each with that child.
__global__ void hetero_expand_kernel(int32_t n_seq, int32_t B, int32_t gamma, int32_t depth,
                                     const int32_t* __restrict__ tok, const uint64_t* __restrict__ key,
                                     const uint64_t* __restrict__ ctx, const uint32_t* __restrict__ pos,
                                     const int32_t* __restrict__ owner, uint64_t* next_key, uint64_t* next_ctx,
                                     uint32_t* next_pos, int32_t* next_owner, int32_t* list_tok, int32_t* list_nd,
                                     int32_t* child_node, uint64_t* node_key, uint64_t* node_ctx,
                                     uint32_t* node_pos) {
    pdl_wait();  // the lists and row ids of the previous launch
    pdl_launch_dependents();
    const int lane = threadIdx.x & 31;
    const int64_t s = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (s >= n_seq) return;
    const int64_t N1 = 1 + (int64_t)B * gamma;
    const int w = depth == 0 ? 1 : B;
    // node lists are numbered depth-major: depth d's start at L_d = n_seq (1 + (d-1) B)
    const int64_t L_d = depth == 0 ? 0 : (int64_t)n_seq * (1 + (int64_t)(depth - 1) * B);
    const int64_t child0 = s * N1 + 1 + (int64_t)depth * B;  // node (s, d+1, 0)
    const int64_t r = s * B + lane;
    int o = -1, x = -1;
    if (lane < B) {
        o = owner[r];
        x = tok[r];
    }
    const bool alive = lane < B && o >= 0 && o < w && x >= 0;
    int first = alive ? lane : -1;
    for (int t = 0; t < B; ++t) {
        const int ot = __shfl_sync(FULL, o, t), xt = __shfl_sync(FULL, x, t);
        const bool at = __shfl_sync(FULL, (int)alive, t) != 0;
        if (alive && at && t < first && ot == o && xt == x) first = t;
    }
    // lane o writes the list of node (s, d, o)
    const int64_t lr = L_d + s * w + lane;
    int m = 0;
    for (int t = 0; t < B; ++t) {
        const int ot = __shfl_sync(FULL, o, t), xt = __shfl_sync(FULL, x, t), ft = __shfl_sync(FULL, first, t);
        const bool at = __shfl_sync(FULL, (int)alive, t) != 0;
        if (lane < w && at && ot == lane && ft == t) {
            list_tok[lr * B + m] = xt;
            child_node[lr * B + m] = (int32_t)(child0 + t);
            ++m;
        }
    }
    if (lane < w) {
        for (int q = m; q < B; ++q) {
            list_tok[lr * B + q] = -1;
            child_node[lr * B + q] = -1;
        }
        list_nd[lr] = m;
    }
    // depth d+1: node (s, d+1, b) is proposal b's when it is the first to reach it
    if (lane < B) {
        uint64_t k = 0, lab = 0;
        uint32_t p = 0;
        if (alive) {
            k = key[r];
            lab = mix64(ctx[r] ^ ((uint64_t)(uint32_t)(x + 1) * 0x9E3779B97F4A7C15ull));
            p = pos[r] + 1u;
        }
        const bool owns = alive && first == lane;
        node_key[child0 + lane] = owns ? k : 0;
        node_ctx[child0 + lane] = owns ? lab : 0;
        node_pos[child0 + lane] = owns ? p : 0u;
        if (depth + 1 < gamma) {
            next_key[r] = k;
            next_ctx[r] = lab;
            next_pos[r] = p;
            next_owner[r] = alive ? first : -1;
        }
    }
}

// block J of the augmented race's winning point (Y, J) for each token
__global__ void hetero_block_kernel(int64_t n, int32_t B, const int32_t* __restrict__ tok,
                                    const uint64_t* __restrict__ key, const uint64_t* __restrict__ ctx,
                                    const uint32_t* __restrict__ pos, int32_t* __restrict__ out) {
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < n; t += (int64_t)gridDim.x * blockDim.x) {
        const int32_t y = tok[t];
        out[t] = y >= 0 ? block_j(word_of(key[t] ^ kBlockJ, ctx[t], pos[t], y, 1), B) : -1;
    }
}

__global__ void words_kernel(const uint64_t* __restrict__ key, const uint64_t* __restrict__ ctx,
                             const uint32_t* __restrict__ pos, int64_t n_rows, int64_t V, int32_t arrival,
                             uint32_t* __restrict__ out) {
    const int64_t total = n_rows * V;
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < total; t += (int64_t)gridDim.x * blockDim.x) {
        int64_t r = t / V, i = t - r * V;
        out[t] = word_of(key[r], ctx[r], pos[r], i, arrival);
    }
}

// largest |x32(w) - log2(-log2 u(w))| over a word range; the fp64 reference
// uses E = -ln u through u for u <= 1/2 and through v = 1 - u above
__global__ void selftest_kernel(uint64_t w0, uint64_t w1, float* out) {
    float worst = 0.0f;
    for (uint64_t w = w0 + (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; w < w1;
         w += (uint64_t)gridDim.x * blockDim.x) {
        uint32_t x = (uint32_t)w;
        float x32 = key_x32(x);
        double xd = log2(exp1_f64(x) * 1.4426950408889634074);
        float d = (float)fabs((double)x32 - xd);
        worst = fmaxf(worst, d);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) worst = fmaxf(worst, __shfl_xor_sync(FULL, worst, o));
    if ((threadIdx.x & 31) == 0) atomicMax(reinterpret_cast<unsigned int*>(out), __float_as_uint(worst));
}

// largest |lg2.approx(x) - log2 x| over the positive fp32 x with bit patterns
// in [b0, b1) (every input of the block key's outer logarithm)
__global__ void selftest_lg2_kernel(uint32_t b0, uint32_t b1, float* out) {
    float worst = 0.0f;
    for (uint64_t b = (uint64_t)b0 + (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; b < b1;
         b += (uint64_t)gridDim.x * blockDim.x) {
        const float x = __uint_as_float((uint32_t)b);
        const float d = (float)fabs((double)lg2_approx(x) - log2((double)x));
        worst = fmaxf(worst, d);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) worst = fmaxf(worst, __shfl_xor_sync(FULL, worst, o));
    if ((threadIdx.x & 31) == 0) atomicMax(reinterpret_cast<unsigned int*>(out), __float_as_uint(worst));
}

// Philox-only throughput: every thread generates blocks c0 = t, t + stride, ...
// with the row-specialised generator of the streaming kernels and folds the
// words into one value, so the kernel is bound by the Philox multiplies alone
// (the ceiling of the race kernels on bf16 rows).
__global__ void __launch_bounds__(256) philox_rate_kernel(uint64_t key, uint64_t ctx, uint32_t pos, uint64_t n_blocks,
                                                          uint32_t* out) {
    RowPhilox rp;
    rp.init(key, ctx, pos);
    uint32_t acc = 0;
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t b = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; b < n_blocks; b += 2 * stride) {
        const uint4 v0 = rp.block((uint32_t)b);
        const uint4 v1 = rp.block((uint32_t)(b + stride));
        acc ^= v0.x ^ v0.y ^ v0.z ^ v0.w ^ v1.x ^ v1.y ^ v1.z ^ v1.w;
    }
    out[(uint64_t)blockIdx.x * blockDim.x + threadIdx.x] = acc;
}

cudaError_t launch_philox_rate(uint64_t n_blocks, uint32_t* out, int out_len, cudaStream_t stream) {
    int blocks = out_len / 256;
    if (blocks < 1) return cudaErrorInvalidValue;
    philox_rate_kernel<<<blocks, 256, 0, stream>>>(0x0123456789abcdefull, 0xfedcba9876543210ull, 7u, n_blocks, out);
    return cudaGetLastError();
}

cudaError_t launch_wm_score(const int32_t* tokens, const uint64_t* key, const uint64_t* ctx, const uint32_t* pos,
                            int64_t n, int32_t n_seg, const int64_t* seg_off, const ScoreParams& P, float* out_score,
                            double* out_sum, double* out_logp, cudaStream_t stream) {
    const int32_t ns = seg_off ? n_seg : 1;
    if (out_sum) {
        cudaError_t e = cudaMemsetAsync(out_sum, 0, sizeof(double) * (size_t)ns, stream);
        if (e != cudaSuccess) return e;
    }
    if (n > 0) {
        // one wave: as many warps as the GPU holds at once, each a contiguous chunk
        // (a multiple of the 128 tokens of one load group)
        const int64_t resident =
            (int64_t)device_sm_count() * resident_ctas(kOccScore, (const void*)wm_score_kernel<true>, 256) * (256 / 32);
        const int64_t group = 32 * kScoreAhead;
        const int64_t chunk = ((n + resident - 1) / resident + group - 1) / group * group;
        const int64_t warps = (n + chunk - 1) / chunk;
        const int64_t blocks = (warps * 32 + 255) / 256;
        // pairs of tuples are loaded and stored together, 16 bytes of keys and labels, 8 of tokens, positions
        // and scores; arrays that all start on 16-byte boundaries take that path (chunks start on multiples
        // of 128 tuples)
        auto al = [](const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; };
        const bool vec = al(tokens) && al(key) && al(ctx) && al(pos) && (out_score == nullptr || al(out_score));
        if (vec)
            wm_score_kernel<true><<<(unsigned)blocks, 256, 0, stream>>>(tokens, key, ctx, pos, n, n_seg, seg_off, P,
                                                                        out_score, out_sum, chunk);
        else
            wm_score_kernel<false><<<(unsigned)blocks, 256, 0, stream>>>(tokens, key, ctx, pos, n, n_seg, seg_off, P,
                                                                         out_score, out_sum, chunk);
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    if (out_logp && ns > 0) {
        seg_logp_kernel<<<(ns + kLogpSegs - 1) / kLogpSegs, 2 * kLogpSegs, 0, stream>>>(n, ns, seg_off, out_sum, P.kind, out_logp);
        return cudaGetLastError();
    }
    return cudaSuccess;
}

cudaError_t launch_tree_expand(int32_t n_seq, int32_t K, int32_t gamma, int32_t depth, const int32_t* tok,
                               const int32_t* mult, const int32_t* ndist, const uint64_t* key, const uint64_t* ctx,
                               const uint32_t* pos, const int32_t* row_k, uint64_t* next_key, uint64_t* next_ctx,
                               uint32_t* next_pos, int32_t* next_k, int32_t* child_node, uint64_t* node_key,
                               uint64_t* node_ctx, uint32_t* node_pos, cudaStream_t stream) {
    if (n_seq == 0) return cudaSuccess;
    const int64_t blocks = ((int64_t)n_seq * 32 + 255) / 256;
    const cudaError_t e = launch_pdl(tree_expand_kernel, dim3((unsigned)blocks), dim3(256), 0, stream, n_seq, K, gamma,
                                     depth, tok, mult, ndist, key, ctx, pos, row_k, next_key, next_ctx, next_pos,
                                     next_k, child_node, node_key, node_ctx, node_pos);
    return e != cudaSuccess ? e : cudaGetLastError();
}

cudaError_t launch_hetero_expand(int32_t n_seq, int32_t B, int32_t gamma, int32_t depth, const int32_t* tok,
                                 const uint64_t* key, const uint64_t* ctx, const uint32_t* pos, const int32_t* owner,
                                 uint64_t* next_key, uint64_t* next_ctx, uint32_t* next_pos, int32_t* next_owner,
                                 int32_t* list_tok, int32_t* list_nd, int32_t* child_node, uint64_t* node_key,
                                 uint64_t* node_ctx, uint32_t* node_pos, cudaStream_t stream) {
    if (n_seq == 0) return cudaSuccess;
    const int64_t blocks = ((int64_t)n_seq * 32 + 255) / 256;
    const cudaError_t e = launch_pdl(hetero_expand_kernel, dim3((unsigned)blocks), dim3(256), 0, stream, n_seq, B,
                                     gamma, depth, tok, key, ctx, pos, owner, next_key, next_ctx, next_pos, next_owner,
                                     list_tok, list_nd, child_node, node_key, node_ctx, node_pos);
    return e != cudaSuccess ? e : cudaGetLastError();
}

cudaError_t launch_hetero_block(int64_t n, int32_t B, const int32_t* tok, const uint64_t* key, const uint64_t* ctx,
                                const uint32_t* pos, int32_t* out, cudaStream_t stream) {
    if (n == 0) return cudaSuccess;
    int64_t blocks = (n + 255) / 256;
    if (blocks > 152 * 16) blocks = 152 * 16;
    hetero_block_kernel<<<(unsigned)blocks, 256, 0, stream>>>(n, B, tok, key, ctx, pos, out);
    return cudaGetLastError();
}

cudaError_t launch_words(const uint64_t* key, const uint64_t* ctx, const uint32_t* pos, int64_t n_rows, int64_t V,
                         int32_t arrival, uint32_t* out, cudaStream_t stream) {
    int64_t total = n_rows * V;
    if (total == 0) return cudaSuccess;
    int64_t blocks = (total + 255) / 256;
    if (blocks > 65535 * 8) blocks = 65535 * 8;
    words_kernel<<<(unsigned)blocks, 256, 0, stream>>>(key, ctx, pos, n_rows, V, arrival, out);
    return cudaGetLastError();
}

cudaError_t launch_selftest(uint64_t w_begin, uint64_t w_end, float* out, cudaStream_t stream) {
    if (w_end <= w_begin) return cudaSuccess;
    uint64_t n = w_end - w_begin;
    uint64_t blocks = (n + 255) / 256;
    if (blocks > 152 * 64) blocks = 152 * 64;
    selftest_kernel<<<(unsigned)blocks, 256, 0, stream>>>(w_begin, w_end, out);
    return cudaGetLastError();
}

cudaError_t launch_selftest_lg2(uint32_t b0, uint32_t b1, float* out, cudaStream_t stream) {
    if (b1 <= b0) return cudaSuccess;
    uint64_t blocks = ((uint64_t)(b1 - b0) + 255) / 256;
    if (blocks > 152 * 64) blocks = 152 * 64;
    selftest_lg2_kernel<<<(unsigned)blocks, 256, 0, stream>>>(b0, b1, out);
    return cudaGetLastError();
}

}  // namespace pps
